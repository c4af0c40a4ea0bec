// psort_radix.cuh -- step 1 (sort each block) as a least-significant-digit
// radix sort of the order keys, for blocks of many tiles.
//
// A segment is one block of one instance (a single sort with one block is one
// segment).  One kernel counts every digit of every segment; then one kernel
// per digit reads the keys tile by tile, groups each tile by the digit in
// shared memory and writes the groups to their places (one read and one write
// of the data per digit, counting included in neither).  A tile learns where
// its groups go by decoupled look-back (Merrill & Garland, "Single-pass
// Parallel Prefix Scan with Decoupled Look-back", 2016): it publishes its
// digit counts, sums the counts of the tiles before it and publishes the sum.
#pragma once

#include "psort_kernels.cuh"

namespace ps {

// ------------------------------------------------------------- digits
// Digit d of a key is its byte d (records: bytes 0..3 of the payload, then
// bytes 0..7 of the key).
template <typename K> struct Rx;
template <> struct Rx<uint32_t> {
    static constexpr int D = 4;
    __device__ static __forceinline__ unsigned dig(uint32_t k, int d) { return __byte_perm(k, 0, 0x4440 | d); }
    // the bytes lo..d of a key, as a value that compares like them
    using M = uint32_t;
    __device__ static M mask(int lo, int d)
    {
        const uint32_t up = d >= 3 ? ~0u : (1u << (8 * (d + 1))) - 1;
        return up & ~((1u << (8 * lo)) - 1);
    }
    __device__ static __forceinline__ bool lt(uint32_t a, uint32_t b, M m) { return (a & m) < (b & m); }
};
template <> struct Rx<uint64_t> {
    static constexpr int D = 8;
    __device__ static __forceinline__ unsigned dig(uint64_t k, int d)
    {
        return __byte_perm((uint32_t)k, (uint32_t)(k >> 32), d) & 255u;
    }
    using M = uint64_t;
    __device__ static M mask(int lo, int d)
    {
        const uint64_t up = d >= 7 ? ~0ull : (1ull << (8 * (d + 1))) - 1;
        return up & ~((1ull << (8 * lo)) - 1);
    }
    __device__ static __forceinline__ bool lt(uint64_t a, uint64_t b, M m) { return (a & m) < (b & m); }
};

// What one segment's passes do: digits dig[0..npass), ascending.
struct RxPlan {
    int npass;
    int lo;        // lowest digit sorted
    uint8_t dig[16];
};

// Device tables and buffers of one radix sort.  Pass 0 reads `first`, pass i
// writes b (i even) or a (i odd); the last pass (which has an odd index)
// writes `last`.
template <typename K> struct RxArgs {
    GBuf<K> first, a, b, last;
    Inst in;
    int64_t n_B;
    int64_t nseg;            // segments (instances x blocks)
    int64_t R;               // tile slots per segment
    int64_t ntiles;          // nseg * R
    K* const* iptr;          // instances in buffers of their own (first, a and last)
    unsigned long long* hist;  // [nseg][D][256]: digit counts, then their exclusive sums
    RxPlan* plan;            // [nseg]
    unsigned* done;          // [nseg]: finished counting chunks
    unsigned* ticket;        // [D]: next tile of each pass
    int64_t chunk;           // keys per counting chunk
    int64_t RC;              // chunk slots per segment
    int min_pass;            // least number of passes (a sort between two buffers needs some)
    bool keep;               // the last pass leaves order keys
};

template <typename K> __device__ __forceinline__ void rx_seg(const RxArgs<K>& A, int64_t seg, int64_t& off, int64_t& len)
{
    const int64_t inst = A.n_B == 1 ? seg : seg / A.n_B, b = seg - inst * A.n_B;
    int64_t bs, be;
    block_bounds(A.in.len(inst), A.n_B, b, bs, be);
    off = A.in.off(inst) + bs;
    len = be - bs;
}
// The segment's part of a buffer.
template <typename K> __device__ __forceinline__ GBuf<K> rx_sub(const GBuf<K>& g, int64_t off, int64_t len)
{
    return GBuf<K>{g.p + off, len};
}

// The first look-back wait that gave up (tile + 1), recorded like an index
// violation; 0 in every correct run.
static __device__ unsigned long long rx_stall;

// ------------------------------------------------------------ counting
// One CTA counts G digits (group blockIdx.y) of one chunk of one segment.
// Shared counters are private to a lane column: counter (digit value v, lane
// l) is half v&1 of word (v/2)*32 + l, so a warp's 32 updates always go to 32
// different banks whatever the keys are (a chunk holds fewer than 2^21 keys,
// so 16 bits per lane suffice).  Bound by those updates (one wavefront per
// digit and 32 keys).  The last chunk of a segment to finish makes its plan
// and turns the counts into exclusive sums.
template <int NT, int G, typename K, int XF>
__global__ void __launch_bounds__(NT) k_rx_count(RxArgs<K> A)
{
    constexpr int D = Rx<K>::D;
    extern __shared__ __align__(16) char smem[];
    uint32_t* cnt = (uint32_t*)smem;  // [G][128][32]
    __shared__ unsigned s_last;
    const int64_t seg = blockIdx.x / A.RC, ch = blockIdx.x - seg * A.RC;
    if (seg >= A.nseg) return;
    int64_t off, len;
    rx_seg(A, seg, off, len);
    const int64_t c0 = ch * A.chunk;
    if (c0 >= len) return;
    const int n = (int)(len - c0 < A.chunk ? len - c0 : A.chunk);
    const int g0 = blockIdx.y * G;
    for (int i = threadIdx.x; i < G * 4096; i += NT) cnt[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const GBuf<K> src = A.iptr ? GBuf<K>{A.iptr[seg] + c0, (int64_t)n} : rx_sub(A.first, off + c0, (int64_t)n);
    auto add = [&](const K& k) {
#pragma unroll
        for (int d = 0; d < G; d++) {
            const unsigned v = Rx<K>::dig(k, g0 + d);
            atomicAdd(&cnt[d * 4096 + ((v >> 1) << 5) + lane], (v & 1) ? 65536u : 1u);
        }
    };
    constexpr int U = 8;
    int i = threadIdx.x;
    for (; i + (U - 1) * NT < n; i += U * NT) {
        K k[U];
#pragma unroll
        for (int u = 0; u < U; u++) k[u] = src.template ldx<XF>(i + u * NT);
#pragma unroll
        for (int u = 0; u < U; u++) add(k[u]);
    }
    for (; i < n; i += NT) add(src.template ldx<XF>(i));
    __syncthreads();
    unsigned long long* h = A.hist + seg * (D * 256);
    for (int r = threadIdx.x; r < G * 128; r += NT) {
        uint32_t lo = 0, hi = 0;
#pragma unroll 8
        for (int l = 0; l < 32; l++) {
            const uint32_t w = cnt[r * 32 + ((l + lane) & 31)];
            lo += w & 0xFFFFu;
            hi += w >> 16;
        }
        if (lo) atomicAdd(&h[g0 * 256 + 2 * r], (unsigned long long)lo);
        if (hi) atomicAdd(&h[g0 * 256 + 2 * r + 1], (unsigned long long)hi);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned parts = (unsigned)((len + A.chunk - 1) / A.chunk) * gridDim.y;
        s_last = atomicAdd(&A.done[seg], 1u) == parts - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // one warp per digit: exclusive sums of its 256 counts; a digit that all
    // keys share is skipped
    __shared__ int s_all[D];
    for (int d = threadIdx.x >> 5; d < D; d += NT / 32) {
        unsigned long long v[8], s = 0;
        bool all = false;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            v[q] = __ldcg(&h[d * 256 + lane * 8 + q]);
            all |= v[q] == (unsigned long long)len;
            s += v[q];
        }
        unsigned long long x = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        x -= s;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            h[d * 256 + lane * 8 + q] = x;
            x += v[q];
        }
        all = __any_sync(0xFFFFFFFFu, all);
        if (lane == 0) s_all[d] = all;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        RxPlan p;
        p.lo = 0;
        int act = 0;
        for (int d = 0; d < D; d++) act += !s_all[d];
        // the passes alternate between two buffers: an even number of them,
        // filled up with digits that change nothing
        int want = act + (act & 1);
        if (want < A.min_pass) want = A.min_pass;
        int fill = want - act;
        p.npass = 0;
        for (int d = 0; d < D; d++) {
            if (s_all[d] && fill <= 0) continue;
            if (s_all[d]) fill--;
            p.dig[p.npass++] = (uint8_t)d;
        }
        A.plan[seg] = p;
    }
}

// ------------------------------------------------------------ scatter
// Look-back words: a count with two flag bits on top (1: the tile's own
// counts, 2: counts of all tiles up to this one).
template <typename CT> struct Lb {
    static constexpr int SH = 8 * (int)sizeof(CT) - 2;
    static constexpr CT OWN = (CT)1 << SH, SUM = (CT)2 << SH, FLAGS = (CT)3 << SH;
    static __device__ __forceinline__ CT ld(const CT* p)
    {
        if constexpr (sizeof(CT) == 8) {
            unsigned long long v;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
            return v;
        } else {
            uint32_t v;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
            return v;
        }
    }
    static __device__ __forceinline__ void st(CT* p, CT v)
    {
        if constexpr (sizeof(CT) == 8)
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((unsigned long long)v) : "memory");
        else
            asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"((uint32_t)v) : "memory");
    }
};

// Shared memory of one pass CTA: the tile's keys grouped by digit, one digit
// table per warp, and every digit's destination.
template <typename K, typename CT, int NT, int E> constexpr size_t rx_smem()
{
    return sizeof(K) * NT * E + (NT / 32) * 1024 + 256 * sizeof(CT) + 64;
}

constexpr unsigned RX_SPINS = 1u << 24;  // looks at one predecessor before a wait gives up

// One digit pass.  Persistent CTAs take tiles in order from a counter, so
// every tile before a waiting one is running or done and the look-back ends.
//
// Ranks inside a tile.  Warp w holds the tile's positions [w*32*E, (w+1)*32*E),
// item j of lane l at w*32*E + j*32 + l.  A warp counts its keys in a table of
// its own, one shared-memory atomic per item, whose old value is the key's
// rank; items of one digit value take a match instead (a 32-fold conflict
// otherwise).  An atomic fixes no order among the lanes of one item, so the
// pass checks what it needs: the keys of every group in ascending order of
// the digits sorted so far (the order of keys that agree in those digits does
// not matter).  The check reads what the store loop reads anyway; a tile that
// fails it is ranked again in lane order (eight ballots per item) and stored
// again to the same places.
//
// Bound by shared-memory wavefronts and their latency (L1 data pipe 72%, 50
// instructions per 32 keys at 2^26 uint32).  Measured at 2^28 uniform keys per
// pass: 0.79 ms for uint32 (2.7 TB/s), 1.20 ms for uint64 (3.6 TB/s).  Ranks by
// ballots alone took 1.37 and 1.76 ms (ALU bound, 97 instructions per 32
// keys), __match_any_sync 2.20 ms, matching through shared-memory OR 0.99 ms;
// the check costs 2-3%.
template <typename K, int XF, typename CT, int NT, int E, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) k_rx_pass(RxArgs<K> A, int slot, CT* lb, CT* lb_next)
{
    constexpr int T = NT * E, W = NT / 32, LB = 8;
    static_assert(NT >= 256, "one thread per digit value");
    extern __shared__ __align__(16) char smem[];
    K* sk = (K*)smem;
    uint32_t* wt = (uint32_t*)(sk + T);  // [W][256]
    CT* gb = (CT*)(wt + W * 256);        // [256]: destination of the digit's group, less its place in the tile
    __shared__ unsigned s_tile, s_w[8];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t* my = wt + w * 256;
    const bool single = A.nseg == 1;
    if (single && slot >= A.plan[0].npass) return;
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(&A.ticket[slot], 1u);
        ((uint4*)my)[lane] = make_uint4(0, 0, 0, 0);
        ((uint4*)my)[lane + 32] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= A.ntiles) return;
        const int64_t seg = single ? 0 : tile / A.R, lt = single ? tile : tile - seg * A.R;
        int64_t off, len;
        rx_seg(A, seg, off, len);
        const int64_t o = lt * T;
        const RxPlan& pl = A.plan[seg];
        if (o >= len || slot >= pl.npass) {
            __syncthreads();
            continue;
        }
        const int d = pl.dig[slot];
        const bool head = slot == 0, tail = slot + 1 == pl.npass;
        const GBuf<K> own = A.iptr ? GBuf<K>{A.iptr[seg], len} : rx_sub(A.a, off, len);
        const GBuf<K> oth = rx_sub(A.b, off, len);
        const GBuf<K> src = head ? (A.iptr ? own : rx_sub(A.first, off, len)) : (slot & 1) ? oth : own;
        const GBuf<K> dst = tail ? (A.iptr ? own : rx_sub(A.last, off, len)) : (slot & 1) ? own : oth;
        const int n = (int)(len - o < T ? len - o : T);
        const bool full = n == T;
        const int p0 = w * 32 * E + lane;
        K k[E];
        uint32_t rk[E];
        auto load = [&]() {
            if (full) {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = src.ld(o + p0 + j * 32);
            } else {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = p0 + j * 32 < n ? src.ld(o + p0 + j * 32) : K(0);
            }
            if (head) {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = xform<XF>(k[j]);
            }
        };
        load();
#pragma unroll
        for (int j = 0; j < E; j++) {
            const unsigned v = Rx<K>::dig(k[j], d);
            int same;
            __match_all_sync(0xFFFFFFFFu, v, &same);
            if (same && full) {
                const uint32_t old = my[v];
                __syncwarp();
                if (lane == 0) my[v] = old + 32;
                __syncwarp();
                rk[j] = old + lane;
            } else if (full || p0 + j * 32 < n) {
                rk[j] = atomicAdd(&my[v], 1u);
            }
        }
        __syncthreads();
        uint32_t tot = 0, ex = 0;
        CT* row = lb + tile * 256;
        if (tid < 256) {
#pragma unroll
            for (int i = 0; i < W; i++) {
                const uint32_t c = wt[i * 256 + tid];
                wt[i * 256 + tid] = tot;
                tot += c;
            }
            const CT start = lt == 0 ? (CT)A.hist[(seg * Rx<K>::D + d) * 256 + tid] : 0;
            if (lt == 0) gb[tid] = start;
            Lb<CT>::st(row + tid, lt == 0 ? (Lb<CT>::SUM | (start + tot)) : (Lb<CT>::OWN | (CT)tot));
            lb_next[tile * 256 + tid] = 0;
            uint32_t x = tot;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, s);
                if (lane >= s) x += y;
            }
            if (lane == 31) s_w[w] = x;
            ex = x - tot;
        }
        __syncthreads();
        if (tid < 256) {
#pragma unroll
            for (int i = 0; i < 7; i++)
                if (i < w) ex += s_w[i];
#pragma unroll
            for (int i = 0; i < W; i++) wt[i * 256 + tid] += ex;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < E; j++)
            if (full || p0 + j * 32 < n) {
                const uint32_t q = my[Rx<K>::dig(k[j], d)] + rk[j];
                if (PS_IN(q, T, 51)) sk[q] = k[j];
            }
        if (tid < 256) {
            CT excl = 0;
            if (lt == 0) {
                excl = gb[tid];
            } else {
                const CT* p = lb + (tile - 1) * 256 + tid;
                int64_t left = lt;  // predecessors not yet summed
                unsigned spins = 0;
                for (bool more = true; more;) {
                    CT v[LB];
#pragma unroll
                    for (int q = 0; q < LB; q++) v[q] = q < left ? Lb<CT>::ld(p - q * 256) : (CT)0;
#pragma unroll
                    for (int q = 0; q < LB; q++) {
                        if (!more) break;
                        if ((v[q] & Lb<CT>::FLAGS) == 0) {
                            if (++spins > RX_SPINS) {
                                atomicExch(&rx_stall, (unsigned long long)tile + 1);
                                more = false;
                            }
                            break;
                        }
                        excl += v[q] & ~Lb<CT>::FLAGS;
                        p -= 256;
                        left--;
                        if (v[q] & Lb<CT>::SUM) more = false;
                    }
                }
                Lb<CT>::st(row + tid, Lb<CT>::SUM | (excl + tot));
            }
            gb[tid] = excl - ex;
        }
        __syncthreads();
        const typename Rx<K>::M m = Rx<K>::mask(pl.lo, d);
        const bool inv = tail && !A.keep;
        auto store = [&]() {
            bool bad = false;
#pragma unroll
            for (int q = 0; q < E; q++) {
                const int i = tid + q * NT;
                if (full || i < n) {
                    const K x = sk[i];
                    if (!head) bad |= Rx<K>::lt(x, sk[i > 0 ? i - 1 : 0], m);
                    const CT p = gb[Rx<K>::dig(x, d)] + (CT)i;
                    // (a stale sum after an abandoned wait must not leave the segment)
                    if (p < (CT)len) {
                        if (inv) dst.template stx<XF>((int64_t)p, x);
                        else dst.st((int64_t)p, x);
                    }
                }
            }
            return bad;
        };
        if (__syncthreads_or(store())) {
#pragma unroll 1
            for (int j = 0; j < E; j++) {
                const int i = p0 + j * 32;
                const K x = i < n ? (head ? src.template ldx<XF>(o + i) : src.ld(o + i)) : K(0);
                const unsigned v = Rx<K>::dig(x, d);
                unsigned mt = __ballot_sync(0xFFFFFFFFu, i < n);
#pragma unroll
                for (int b = 0; b < 8; b++) {
                    const bool bit = (v >> b) & 1;
                    const unsigned u = __ballot_sync(0xFFFFFFFFu, bit);
                    mt &= bit ? u : ~u;
                }
                const unsigned r = __popc(mt & ((1u << lane) - 1));
                const uint32_t old = my[v];
                __syncwarp();
                if (i < n) {
                    if (r == 0) my[v] = old + __popc(mt);
                    if (PS_IN(old + r, T, 52)) sk[old + r] = x;
                }
                __syncwarp();
            }
            __syncthreads();
            store();
            __syncthreads();
        }
    }
}

}  // namespace ps

// psort_radix.cuh -- step 1 (sort each block) as a least-significant-digit
// radix sort of the order keys, for blocks of many tiles.
//
// A segment is one instance, sorted as one block (a single sort is one segment).
// One kernel counts every digit of every segment; then one kernel per digit reads
// the keys tile by tile, groups each tile by the digit in shared memory and writes
// the groups to their places (one read and one write of the data per digit,
// counting included in neither).  A tile learns where its groups go by decoupled
// look-back (Merrill & Garland, "Single-pass Parallel Prefix Scan with Decoupled
// Look-back", 2016): it publishes its digit counts, sums the counts of the tiles
// before it and publishes the sum.
#pragma once

#include <type_traits>

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
    __device__ static __forceinline__ bool same(uint32_t a, uint32_t b, M m) { return ((a ^ b) & m) == 0; }
    __device__ static __forceinline__ uint64_t word(uint32_t a, M m) { return a & m; }
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
    __device__ static __forceinline__ bool same(uint64_t a, uint64_t b, M m) { return ((a ^ b) & m) == 0; }
    __device__ static __forceinline__ uint64_t word(uint64_t a, M m) { return a & m; }
};

template <> struct Rx<Rec> {
    static constexpr int D = 12;
    __device__ static __forceinline__ unsigned dig(const Rec& r, int d)
    {
        return d < 4 ? __byte_perm(r.p, 0, 0x4440 | d) : Rx<uint64_t>::dig(r.k, d - 4);
    }
    struct M {
        uint64_t k;
        uint32_t p;
    };
    __device__ static M mask(int lo, int d)
    {
        return M{d < 4 ? 0 : Rx<uint64_t>::mask(lo < 4 ? 0 : lo - 4, d - 4),
                 lo > 3 ? 0 : Rx<uint32_t>::mask(lo, d > 3 ? 3 : d)};
    }
    __device__ static __forceinline__ bool lt(const Rec& a, const Rec& b, M m)
    {
        return (a.k & m.k) < (b.k & m.k) || ((a.k & m.k) == (b.k & m.k) && (a.p & m.p) < (b.p & m.p));
    }
    __device__ static __forceinline__ bool same(const Rec& a, const Rec& b, M m)
    {
        return ((a.k ^ b.k) & m.k) == 0 && ((a.p ^ b.p) & m.p) == 0;
    }
    __device__ static __forceinline__ uint64_t word(const Rec& a, M m)
    {
        return (a.k & m.k) + (uint64_t)(a.p & m.p) * 0x9E3779B97F4A7C15ull;
    }
};

// Keys of one tile in shared memory.
template <typename K> struct RxTile {
    K* a;
    static constexpr size_t bytes(int n) { return sizeof(K) * n; }
    __device__ RxTile(char*& sp, int n) : a((K*)sp) { sp += bytes(n); }
    __device__ __forceinline__ K ld(int i) const { return a[i]; }
    __device__ __forceinline__ void st(int i, const K& v) const { a[i] = v; }
};
template <> struct RxTile<Rec> {
    uint64_t* k;
    uint32_t* p;
    static constexpr size_t bytes(int n) { return 12 * (size_t)n; }
    __device__ RxTile(char*& sp, int n) : k((uint64_t*)sp), p((uint32_t*)(sp + 8 * (size_t)n)) { sp += bytes(n); }
    __device__ __forceinline__ Rec ld(int i) const { return Rec{k[i], p[i]}; }
    __device__ __forceinline__ void st(int i, const Rec& v) const
    {
        k[i] = v.k;
        p[i] = v.p;
    }
};

// What one segment's passes do: digits dig[0..npass), ascending.
struct RxPlan {
    int npass;
    int lo;        // lowest digit sorted
    uint8_t dig[16];
};

// Where a segment's work lies: its first tile, counting chunk and fix tile
// among those of all segments, and its sample.
struct RxSegAt {
    int tile0, chunk0, fix0;
    int S;         // sampled keys (0: none, every digit is sorted)
    int b0;        // leading bytes of the sample's first choice
    int64_t tab0;  // its hash tables
};
// Work of k_rx_long: positions [s, e) of a segment.
struct RxBad {
    int64_t s, e;
    int seg;
    int tile;                 // 1: the runs inside one fix tile, 0: one run that spans tiles
    unsigned slot;            // its first row of the digit table (runs longer than LONG_ONE)
    unsigned ticket, done;    // tasks taken and finished (the same)
    unsigned dp;              // bits that differ among its payloads and keys (the same)
    unsigned long long dk;
};
// Device tables and buffers of one radix sort.  Pass 0 reads a, pass i writes b (i
// even) or a (i odd).  (A last pass of even index leaves the keys in b: only when
// low digits were left out, k_rx_fix then moves them to a.)
// (first and last are a, for the digit passes: with a in their places, or the members
// in the order of the kernels that read them, the passes have the same registers and
// spills but take up to 0.8% longer: 2^26 float64 2128 against 2111 us a sort.)
template <typename K> struct RxArgs {
    GBuf<K> first, a, b, last;
    Inst in;
    int64_t nseg;            // segments (instances)
    K* const* iptr;          // instances in buffers of their own, in place of a
    unsigned long long* hist;  // [nseg][D][256]: digit counts, then their exclusive sums
    RxPlan* plan;            // [nseg]
    unsigned* done;          // [nseg]: finished counting chunks
    unsigned* ticket;        // [D]: next tile of each pass
    int T;                   // keys per tile of a digit pass
    int64_t chunk;           // keys per counting chunk
    // one segment: its numbers; several (k_rx_at): tables of them
    RxSegAt one;
    int64_t ntiles1;
    RxSegAt* at;             // [nseg]
    int *tile_seg, *chunk_seg, *fix_seg;  // the segment of every tile, chunk and fix tile
    int64_t* total;          // tiles, chunks, fix tiles
    int* maxpass;            // most passes of any segment
    bool sampled;            // 64-bit keys and records: choose digits by sample
    unsigned* descents;      // records: set if the payloads do not ascend
    unsigned* hits;          // [nseg][RX_TRY]: the sample's hits per choice of the lowest digit
    unsigned* tab;           // hash tables
    uint8_t* flags;          // [fix tiles], see k_rx_fix; LISTED: the long run that starts there is listed
    unsigned* nflag;         // number of flagged tiles
    RxBad* bad;              // [2 * fix tiles]: k_rx_long's list
    unsigned* bads;          // [4]: its entries, rows of dtab given out; listing tasks taken and finished
    void* dtab;              // digit table, 256 counts a row (CT)
    unsigned rows;           // of dtab
    unsigned spins;          // looks in vain, over a tile's look-back or at a count, before the wait gives up
    unsigned* err;           // set when one gave up (host memory, where someone waits for the sort)
    bool keep;               // the last pass leaves order keys
};
constexpr int FT = 4096;  // positions of a fix tile (k_rx_fix)

template <typename K> __device__ __forceinline__ void rx_seg(const RxArgs<K>& A, int64_t seg, int64_t& off, int64_t& len)
{
    off = A.in.off(seg);
    len = A.in.len(seg);
}
// The segment's part of a buffer.
template <typename K> __device__ __forceinline__ GBuf<K> rx_sub(const GBuf<K>& g, int64_t off, int64_t len)
{
    return GBuf<K>{g.p + off, len};
}
template <> __device__ __forceinline__ GBuf<Rec> rx_sub(const GBuf<Rec>& g, int64_t off, int64_t len)
{
    return GBuf<Rec>{g.k + off, g.p + off, len};
}
// The segment's part of its instance's own buffer (keys only).
template <typename K> __device__ __forceinline__ GBuf<K> rx_own(K* const* iptr, int64_t seg, int64_t off, int64_t len)
{
    return GBuf<K>{iptr[seg] + off, len};
}
template <> __device__ __forceinline__ GBuf<Rec> rx_own(Rec* const*, int64_t, int64_t, int64_t) { return GBuf<Rec>{nullptr, nullptr, 0}; }
// Tells the compiler that a buffer whose address it has not seen as a kernel
// argument lies in device memory (its loads then need not wait for stores to
// shared memory).
template <typename K> __device__ __forceinline__ GBuf<K> rx_global(const GBuf<K>& b)
{
    __builtin_assume(__isGlobal(b.p));
    return b;
}
template <> __device__ __forceinline__ GBuf<Rec> rx_global(const GBuf<Rec>& b)
{
    __builtin_assume(__isGlobal(b.k));
    __builtin_assume(__isGlobal(b.p));
    return b;
}
// A key of which only the digits of group g0.. matter.
template <int XF, typename K> __device__ __forceinline__ K rx_ld_digits(const GBuf<K>& b, int64_t i, int) { return b.template ldx<XF>(i); }
template <int XF> __device__ __forceinline__ Rec rx_ld_digits(const GBuf<Rec>& b, int64_t i, int g0)
{
    if (!PS_IN(i, b.n, 1)) return Rec{0, 0};
    return g0 < 4 ? Rec{0, b.p[i]} : Rec{b.k[i], 0};
}

// The first wait that gave up (its tile + 1), recorded like an index violation;
// 0 in every correct run.
static __device__ unsigned long long rx_stall;
// A wait gave up: the result is wrong, and whoever waits for the sort is told.  (The
// kernels after it stay inside their buffers whatever order the keys are in.)
template <typename K> __device__ __forceinline__ void rx_give_up(const RxArgs<K>& A, unsigned long long what)
{
    atomicExch(&rx_stall, what + 1);
    *(volatile unsigned*)A.err = 1;
}

// ------------------------------------------------------------ sampling
// How many low bytes the passes may leave out (64-bit keys and records).
// Sorting by the leading bytes alone leaves runs of keys that agree in them;
// where such runs are short, putting them in order afterwards (k_rx_fix) costs
// less than the passes it saves: 2^30 uniform 64-bit keys are nearly distinct
// in their leading four bytes.  The sample tells: S keys at hashed positions
// enter one hash table per choice of `lo` (open addressing, keyed by the bytes
// lo and above); a key that meets an earlier, different one of the same leading
// bytes counts as a hit.  S keys have S^2/2 pairs, so a key has about
// 2 * hits * n / S^2 different ones in its run; the smallest number of leading
// bytes that keeps this at RX_RUN or less wins.  Hits count whatever order
// the two keys come in: nearly sorted input has long runs too.  A guess can be
// wrong (one value makes up a large share of the input and few of its
// neighbours share its leading bytes: the sample sees none of them); it then
// costs the passes of k_rx_long, never order.  Measured: 2^30 int64 uniform 47.4 -> 27.3 ms, 2^26
// float64 Gaussian 3.03 -> 2.3 ms (five leading bytes), a copy of the keys
// included.
// Records of equal keys differ in their payload.  Where the payloads ascend
// over the whole input (the position, in an argsort) the passes over the key
// leave them in order, and such pairs are no hits.
// The choices are RX_TRY numbers of leading bytes from the fewest that could
// tell as many uniform keys apart.
constexpr int RX_RUN = 1;
constexpr int RX_SAMPLE_MAX = 1 << 16, RX_TRY = 4, RX_SLOTS = 4;  // (table slots per sampled key)
// sqrt(8 n) sampled keys: runs with one other key each then give four hits.
__host__ __device__ inline int rx_samples(int64_t n)
{
    int s = 128;
    while (s < RX_SAMPLE_MAX && (int64_t)s * s < 8 * n) s *= 2;
    return s;
}
__host__ __device__ inline int rx_lead(int64_t n)
{
    int b = 1;
    while (b < 8 && (int64_t(1) << (8 * b)) < n) b++;
    return b;
}
__device__ __forceinline__ uint64_t rx_mix(uint64_t z)
{
    // SplitMix64's finaliser (Steele, Lea & Flood 2014)
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
template <typename K> __device__ __forceinline__ RxSegAt rx_at(const RxArgs<K>& A, int64_t seg)
{
    return A.nseg == 1 ? A.one : A.at[seg];
}
template <typename K> __device__ __forceinline__ bool rx_differ(const K& x, const K& y, bool) { return x != y; }
template <> __device__ __forceinline__ bool rx_differ(const Rec& x, const Rec& y, bool ascending)
{
    return x.k != y.k || (!ascending && x.p != y.p);
}
// Whether the payloads of records ascend: sets *descents if one does not (the
// other CTAs then stop looking).
template <int NT> __global__ void __launch_bounds__(NT) k_rx_descents(const uint32_t* p, int64_t n, unsigned* descents)
{
    kernel_entry();
    constexpr int U = 8;
    for (int64_t i0 = (int64_t)blockIdx.x * NT * U; i0 < n; i0 += (int64_t)gridDim.x * NT * U) {
        if (__syncthreads_or(*(volatile unsigned*)descents != 0)) return;
        bool down = false;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = i0 + u * NT + threadIdx.x;
            if (i > 0 && i < n) down |= p[i] < p[i - 1];
        }
        if (__syncthreads_or(down)) {
            if (threadIdx.x == 0) *descents = 1;
            return;
        }
    }
}
// CTA (segment, choice, part of the sample); tab: [RX_TRY][RX_SLOTS * S] entries per
// segment, sample + 1 in 17 bits and 15 further bits of the hash above them, so that
// a probe reads another sample only when it is likely the same prefix.  Bound by the
// longest chain of probes in a warp, an L2 round trip each (2^20 keys: 20 -> 5 us of kernel;
// two slots per key and no hash bits took twice the probes, each with a read of the
// other key).
template <typename K, int XF>
__global__ void __launch_bounds__(128) k_rx_sample(RxArgs<K> A)
{
    kernel_entry();
    constexpr int D = Rx<K>::D;
    const int64_t seg = blockIdx.x;
    const RxSegAt at = rx_at(A, seg);
    const int S = at.S, lo = D - at.b0 - (int)blockIdx.y;
    if (lo < 1) return;
    int64_t off, n;
    rx_seg(A, seg, off, n);
    const GBuf<K> src = A.iptr ? rx_own(A.iptr, seg, 0, n) : rx_sub(A.a, off, n);
    auto pos = [&](int j) { return (int64_t)__umul64hi(rx_mix((uint64_t)(j + 1) * 0x9E3779B97F4A7C15ull), (uint64_t)n); };
    const typename Rx<K>::M m = Rx<K>::mask(lo, D - 1);
    const bool asc = *A.descents == 0;
    const unsigned slots = RX_SLOTS * (unsigned)S;
    unsigned* t = A.tab + at.tab0 + (size_t)blockIdx.y * slots;
    unsigned c = 0;
    for (int i = blockIdx.z * 128 + threadIdx.x; i < S; i += gridDim.z * 128) {
        const int64_t pi = pos(i);
        const K x = src.template ldx<XF>(pi);
        const uint64_t h = rx_mix(Rx<K>::word(x, m));
        const unsigned tag = (unsigned)(h >> 49);
        unsigned q = (unsigned)h & (slots - 1);
        for (unsigned probe = 0; probe < slots; probe++) {
            const unsigned cur = atomicCAS(&t[q], 0u, (tag << 17) | (unsigned)(i + 1));
            if (cur == 0) break;
            if ((cur >> 17) == tag) {
                const K y = src.template ldx<XF>(pos((int)(cur & 0x1FFFFu) - 1));
                if (Rx<K>::same(x, y, m)) {
                    c += rx_differ(x, y, asc);
                    break;
                }
            }
            q = (q + 1) & (slots - 1);
        }
    }
    c = __reduce_add_sync(0xFFFFFFFFu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&A.hits[seg * RX_TRY + blockIdx.y], c);
}
// The choice, by one warp: the first number of leading bytes with few enough hits.
template <typename K> __device__ __forceinline__ int rx_choose_lo(const RxArgs<K>& A, int64_t seg, const RxSegAt& at, int64_t n)
{
    constexpr int D = Rx<K>::D;
    if (at.S == 0) return 0;
    const int q = threadIdx.x & 31;
    const double h = q < RX_TRY ? (double)__ldcg(&A.hits[seg * RX_TRY + q]) : 0.0;
    const bool ok = q < RX_TRY && h * 2.0 * (double)n <= (double)RX_RUN * (double)at.S * (double)at.S;
    const unsigned b = __ballot_sync(0xFFFFFFFFu, ok);
    const int lo = b ? D - at.b0 - (__ffs(b) - 1) : 0;
    return lo < 0 ? 0 : lo;
}

// ------------------------------------------------------------ several segments
// Numbers every segment's tiles, counting chunks, fix tiles and hash tables
// (one CTA), then lists the segment of each (a warp per segment).
template <int NT, typename K> __global__ void __launch_bounds__(NT) k_rx_at(RxArgs<K> A)
{
    kernel_entry();
    const int64_t per = (A.nseg + NT - 1) / NT, s0 = threadIdx.x * per, s1 = s0 + per < A.nseg ? s0 + per : A.nseg;
    int64_t c[4] = {0, 0, 0, 0};
    auto sizes = [&](int64_t seg, int64_t (&v)[4]) {
        int64_t off, n;
        rx_seg(A, seg, off, n);
        if (n < 0) n = 0;
        v[0] = (n + A.T - 1) / A.T;
        v[1] = (n + A.chunk - 1) / A.chunk;
        v[2] = A.sampled ? (n + FT - 1) / FT : 0;
        v[3] = A.sampled ? RX_TRY * RX_SLOTS * (int64_t)rx_samples(n) : 0;
        return n;
    };
    for (int64_t seg = s0; seg < s1; seg++) {
        int64_t v[4];
        sizes(seg, v);
        for (int q = 0; q < 4; q++) c[q] += v[q];
    }
    for (int q = 0; q < 4; q++) {
        int64_t tot;
        c[q] = block_exscan<NT>(c[q], &tot);
        if (threadIdx.x == 0 && q < 3) A.total[q] = tot;
    }
    for (int64_t seg = s0; seg < s1; seg++) {
        int64_t v[4];
        const int64_t n = sizes(seg, v);
        A.at[seg] = RxSegAt{(int)c[0], (int)c[1], (int)c[2], A.sampled ? rx_samples(n) : 0, rx_lead(n), c[3]};
        for (int q = 0; q < 4; q++) c[q] += v[q];
    }
}
template <typename K> __global__ void __launch_bounds__(256) k_rx_lists(RxArgs<K> A)
{
    kernel_entry();
    const int64_t seg = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (seg >= A.nseg) return;
    const RxSegAt at = A.at[seg];
    int64_t off, n;
    rx_seg(A, seg, off, n);
    const int lane = threadIdx.x & 31;
    for (int64_t i = lane; i * A.T < n; i += 32) A.tile_seg[at.tile0 + i] = (int)seg;
    for (int64_t i = lane; i * A.chunk < n; i += 32) A.chunk_seg[at.chunk0 + i] = (int)seg;
    if (A.sampled)
        for (int64_t i = lane; i * FT < n; i += 32) A.fix_seg[at.fix0 + i] = (int)seg;
}

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
    kernel_entry();
    constexpr int D = Rx<K>::D;
    extern __shared__ __align__(16) char smem[];
    uint32_t* cnt = (uint32_t*)smem;  // [G][128][32]
    __shared__ unsigned s_last;
    if (A.nseg > 1 && blockIdx.x >= A.total[1]) return;
    const int64_t seg = A.nseg == 1 ? 0 : A.chunk_seg[blockIdx.x];
    const RxSegAt at = rx_at(A, seg);
    const int64_t ch = blockIdx.x - at.chunk0;
    int64_t off, len;
    rx_seg(A, seg, off, len);
    const int64_t c0 = ch * A.chunk;
    if (c0 >= len) return;
    const int n = (int)(len - c0 < A.chunk ? len - c0 : A.chunk);
    const int g0 = blockIdx.y * G;
    const int lo0 = D > G ? rx_choose_lo(A, seg, at, len) : 0;
    if (g0 + G <= lo0) return;
    for (int i = threadIdx.x; i < G * 4096; i += NT) cnt[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const GBuf<K> src = rx_global(A.iptr ? rx_own(A.iptr, seg, c0, (int64_t)n) : rx_sub(A.a, off + c0, (int64_t)n));
    auto add = [&](const K& k) {
#pragma unroll
        for (int d = 0; d < G; d++) {
            if (D > G && g0 + d < lo0) continue;
            const unsigned v = Rx<K>::dig(k, g0 + d);
            atomicAdd(&cnt[d * 4096 + ((v >> 1) << 5) + lane], (v & 1) ? 65536u : 1u);
        }
    };
    int i = threadIdx.x;
    if constexpr (sizeof(K) <= 8) {
        // 16-byte loads where the chunk is aligned, 8 or 2 in flight (2^28 keys, one
        // by one / 2 / 4 / 8: uint32 456 / 415 / 384 / 360 us, uint64 474 / 447 / 560 / 578)
        if (((uintptr_t)src.p & 15) == 0) {
            constexpr int V = 16 / (int)sizeof(K), U = sizeof(K) == 4 ? 8 : 2;
            const uint4* q = (const uint4*)src.p;
            const int nv = n / V;
            int v0 = 0;  // (the same number of rounds for every thread)
            for (; v0 + U * NT <= nv; v0 += U * NT) {
                uint4 x[U];
#pragma unroll
                for (int u = 0; u < U; u++) x[u] = __ldcs(q + v0 + u * NT + threadIdx.x);
#pragma unroll
                for (int u = 0; u < U; u++) {
                    K k[V];
                    memcpy(k, &x[u], 16);
#pragma unroll
                    for (int v = 0; v < V; v++) add(xform<XF>(k[v]));
                }
            }
            i += v0 * V;  // the rest one by one
        }
    }
    constexpr int U = 8;
    for (; i + (U - 1) * NT < n; i += U * NT) {
        K k[U];
#pragma unroll
        for (int u = 0; u < U; u++) k[u] = rx_ld_digits<XF>(src, i + u * NT, g0);
#pragma unroll
        for (int u = 0; u < U; u++) add(k[u]);
    }
    for (; i < n; i += NT) add(rx_ld_digits<XF>(src, i, g0));
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
        const unsigned parts = (unsigned)((len + A.chunk - 1) / A.chunk) * (gridDim.y - lo0 / G);
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
        p.lo = lo0;
        int act = 0;
        for (int d = lo0; d < D; d++) act += !s_all[d];
        // the passes alternate between two buffers: an even number of them,
        // filled up with digits that change nothing, unless k_rx_fix can move
        // the keys
        int want = lo0 ? act : act + (act & 1);
        if (A.keep && want < 2) want = 2;  // (they also turn the keys into order keys)
        int fill = want - act;
        p.npass = 0;
        for (int d = lo0; d < D; d++) {
            if (s_all[d] && fill <= 0) continue;
            if (s_all[d]) fill--;
            p.dig[p.npass++] = (uint8_t)d;
        }
        A.plan[seg] = p;
        atomicMax(A.maxpass, p.npass);
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

// One segment's part in one pass.
template <typename K> struct RxSegPass {
    GBuf<K> src, dst;
    int64_t len;
    typename Rx<K>::M m, mb;  // the digits sorted after this pass, and before it
    int npass, d, tile0;
    bool inv;  // the pass writes the keys as the user sees them
};
// Records sorted by key bytes only, payloads ascending: a pass has to keep the
// payloads of equal keys in order, so its check looks at them too.
template <typename M> __device__ __forceinline__ void rx_keep_ties(M&, M&, bool) {}
template <> __device__ __forceinline__ void rx_keep_ties(Rx<Rec>::M& m, Rx<Rec>::M& mb, bool ties)
{
    if (ties) m.p = mb.p = ~0u;
}
template <typename K>
__device__ __forceinline__ void rx_seg_pass(const RxArgs<K>& A, int64_t seg, int slot, RxSegPass<K>& sg)
{
    int64_t off, len;
    rx_seg(A, seg, off, len);
    const RxPlan& pl = A.plan[seg];
    sg.len = len;
    sg.tile0 = rx_at(A, seg).tile0;
    sg.npass = len > 0 ? pl.npass : 0;
    if (slot >= sg.npass) return;
    const int d = pl.dig[slot];
    const GBuf<K> own = A.iptr ? rx_own(A.iptr, seg, 0, len) : rx_sub(A.a, off, len);
    const GBuf<K> oth = rx_sub(A.b, off, len);
    sg.d = d;
    const bool tail = slot + 1 == sg.npass;
    sg.src = slot == 0 ? (A.iptr ? own : rx_sub(A.first, off, len)) : (slot & 1) ? oth : own;
    sg.dst = !(slot & 1) ? oth : (tail && !A.iptr) ? rx_sub(A.last, off, len) : own;
    sg.inv = tail && !A.keep;
    sg.m = Rx<K>::mask(pl.lo, d);
    sg.mb = d > pl.lo ? Rx<K>::mask(pl.lo, d - 1) : typename Rx<K>::M{};
    rx_keep_ties(sg.m, sg.mb, pl.lo >= 4 && *A.descents == 0);
}

// Shared memory of one pass CTA: the tile's keys grouped by digit, one digit
// table per warp, and every digit's destination.
template <typename K, typename CT, int NT, int E> constexpr size_t rx_smem()
{
    return RxTile<K>::bytes(NT * E) + (NT / 32) * 1024 + 256 * sizeof(CT) + 64;
}

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
// pass: 0.77 ms for uint32 (2.8 TB/s), 1.10 ms for uint64 (3.9 TB/s), 1.7 ms for
// records (3.8 TB/s).  What a tile costs whatever it holds is kept small: its
// number is fetched ahead, the segment's constants sit in shared memory and ranks
// two to a register (all of them in registers spilled: 1.04 ms for uint32).  Ranks by
// ballots alone took 1.37 and 1.76 ms (ALU bound, 97 instructions per 32
// keys), __match_any_sync 2.20 ms, matching through shared-memory OR 0.99 ms;
// the check costs 2-3%.
template <typename K, int XF, typename CT, int NT, int E, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) k_rx_pass(RxArgs<K> A, int slot, CT* lb, CT* lb_next)
{
    kernel_entry();
    constexpr int T = NT * E, W = NT / 32, LB = 8;
    static_assert(NT >= 256, "one thread per digit value");
    extern __shared__ __align__(16) char smem[];
    char* sp = smem;
    const RxTile<K> sk(sp, T);
    uint32_t* wt = (uint32_t*)sp;        // [W][256]
    CT* gb = (CT*)(wt + W * 256);        // [256]: destination of the digit's group, less its place in the tile
    __shared__ unsigned s_tile, s_w[8];
    __shared__ __align__(16) char s_seg[sizeof(RxSegPass<K>)];
    RxSegPass<K>& sg = *(RxSegPass<K>*)s_seg;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t* my = wt + w * 256;
    const bool single = A.nseg == 1, head = slot == 0;
    if (slot >= *A.maxpass) return;
    if (tid == 0) s_tile = atomicAdd(&A.ticket[slot], 1u);
    __syncthreads();
    int64_t cur = -1;
    const int64_t ntiles = single ? A.ntiles1 : A.total[0];
    for (int64_t tile = s_tile; tile < ntiles;) {
        const int64_t seg = single ? 0 : A.tile_seg[tile];
        if (seg != cur) {
            cur = seg;
            __syncthreads();
            if (tid == 0) rx_seg_pass(A, seg, slot, sg);
            __syncthreads();
        }
        const int64_t lt = tile - sg.tile0, o = lt * T;
        if (slot >= sg.npass || o >= sg.len) {
            __syncthreads();
            if (tid == 0) s_tile = atomicAdd(&A.ticket[slot], 1u);
            __syncthreads();
            tile = s_tile;
            continue;
        }
        const int d = sg.d;
        // the next tile's number, fetched while this tile is ranked
        unsigned next = 0;
        if (tid == NT - 1) next = atomicAdd(&A.ticket[slot], 1u);
        ((uint4*)my)[lane] = make_uint4(0, 0, 0, 0);
        ((uint4*)my)[lane + 32] = make_uint4(0, 0, 0, 0);
        __syncwarp();
        const int n = (int)(sg.len - o < T ? sg.len - o : T);
        const bool full = n == T;
        const int p0 = w * 32 * E + lane;
        K k[E];
        uint32_t rk[E / 2] = {};  // two ranks a register
        auto put_rank = [&](int j, uint32_t r) { rk[j / 2] = (j & 1) ? __byte_perm(rk[j / 2], r, 0x5410) : r; };
        auto load = [&]() {
            const GBuf<K> src = rx_global(sg.src);
            if (full) {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = src.ld(o + p0 + j * 32);
            } else {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = p0 + j * 32 < n ? src.ld(o + p0 + j * 32) : K{};
            }
            if (head) {
#pragma unroll
                for (int j = 0; j < E; j++) k[j] = xform<XF>(k[j]);
            }
        };
        load();
        // Items of one digit value come in crowds (sorted input, few values): a
        // warp looks at four of its items and takes the careful path for all of
        // them if one is uniform.
        bool crowd = !full;
#pragma unroll
        for (int j = 0; j < E; j += E / 4) {
            int s;
            __match_all_sync(0xFFFFFFFFu, Rx<K>::dig(k[j], d), &s);
            crowd |= s != 0;
        }
        if (!crowd) {
#pragma unroll
            for (int j = 0; j < E; j++) put_rank(j, atomicAdd(&my[Rx<K>::dig(k[j], d)], 1u));
        } else {
#pragma unroll
            for (int j = 0; j < E; j++) {
                const unsigned v = Rx<K>::dig(k[j], d);
                int s;
                __match_all_sync(0xFFFFFFFFu, v, &s);
                uint32_t r = 0;
                if (full && s) {
                    r = my[v] + lane;
                    __syncwarp();
                    if (lane == 0) my[v] = r + 32;
                    __syncwarp();
                } else if (full || p0 + j * 32 < n) {
                    r = atomicAdd(&my[v], 1u);
                }
                put_rank(j, r);
            }
        }
        __syncthreads();
        if (tid == NT - 1) s_tile = next;
        uint32_t tot = 0, ex = 0;
        CT* row = lb + tile * 256;
        if (tid < 256) {
#pragma unroll
            for (int i = 0; i < W; i++) tot += wt[i * 256 + tid];
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
            uint32_t at = ex;
#pragma unroll
            for (int i0 = 0; i0 < W; i0 += 4) {
                uint32_t c[4];
#pragma unroll
                for (int i = 0; i < 4; i++) c[i] = wt[(i0 + i) * 256 + tid];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    wt[(i0 + i) * 256 + tid] = at;
                    at += c[i];
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < E; j += 2)
            rk[j / 2] += my[Rx<K>::dig(k[j], d)] + (my[Rx<K>::dig(k[j + 1], d)] << 16);
#pragma unroll
        for (int j = 0; j < E; j++) {
            const uint32_t q = (j & 1) ? rk[j / 2] >> 16 : rk[j / 2] & 0xFFFFu;
            if ((full || p0 + j * 32 < n) && PS_IN(q, T, 51)) sk.st(q, k[j]);
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
                            if (++spins > A.spins) {
                                rx_give_up(A, (unsigned long long)tile);
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
        const unsigned after = s_tile;
        // The tile arrives in the order of the digits before this one: when its
        // first and last key agree in them, all its keys do and any order within
        // a group is right.
        const bool check = (!head || sizeof(K) > 8) && !Rx<K>::same(rx_global(sg.src).ld(o), rx_global(sg.src).ld(o + n - 1), sg.mb);
        // (a stale sum after an abandoned wait must not leave the segment)
        auto store_as = [&](auto ordered, auto inverse) {
            constexpr int U = sizeof(K) == 4 ? 8 : sizeof(K) == 8 ? 4 : 2;  // store batch
            static_assert(E % U == 0, "keys per thread are a multiple of the store batch");
            bool bad = false;
            const GBuf<K> dst = rx_global(sg.dst);
            const typename Rx<K>::M m = sg.m;
            const CT len = (CT)sg.len;
#pragma unroll
            for (int q0 = 0; q0 < E; q0 += U) {
                K x[U], y[U];
                CT p[U];
#pragma unroll
                for (int q = 0; q < U; q++) {
                    const int i = tid + (q0 + q) * NT;
                    const bool in = full || i < n;
                    x[q] = sk.ld(in ? i : 0);
                    if constexpr (decltype(ordered)::value) y[q] = sk.ld(in && i > 0 ? i - 1 : 0);
                }
#pragma unroll
                for (int q = 0; q < U; q++) p[q] = gb[Rx<K>::dig(x[q], d)] + (CT)(tid + (q0 + q) * NT);
#pragma unroll
                for (int q = 0; q < U; q++) {
                    if (!full && tid + (q0 + q) * NT >= n) continue;
                    if constexpr (decltype(ordered)::value) bad |= Rx<K>::lt(x[q], y[q], m);
                    if (p[q] < len) {
                        if constexpr (decltype(inverse)::value) dst.template stx<XF>((int64_t)p[q], x[q]);
                        else dst.st((int64_t)p[q], x[q]);
                    }
                }
            }
            return bad;
        };
        auto store = [&]() {
            const bool inv = sg.inv;
            if (!check) return inv ? store_as(std::false_type{}, std::true_type{}) : store_as(std::false_type{}, std::false_type{});
            return inv ? store_as(std::true_type{}, std::true_type{}) : store_as(std::true_type{}, std::false_type{});
        };
        const bool bad = store();
        if (check && __syncthreads_or(bad)) {
#pragma unroll 1
            for (int j = 0; j < E; j++) {
                const int i = p0 + j * 32;
                const K x = i < n ? (head ? sg.src.template ldx<XF>(o + i) : sg.src.ld(o + i)) : K{};
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
                    if (PS_IN(old + r, T, 52)) sk.st(old + r, x);
                }
                __syncwarp();
            }
            __syncthreads();
            store();
            __syncthreads();
        }
        tile = after;
    }
}

// ------------------------------------------------------- left-out digits
// After passes over the digits lo and above, keys that agree in them stand in
// runs, in an order that the low digits have not had a say in.  One CTA owns
// the runs that start in its FT positions.  It lists them (most keys are runs
// of their own and need nothing more), one thread sorts each listed run of at
// most FL keys by insertion in shared memory, and runs that changed are
// written back.  Keys of a run all stay inside it, so the leading bytes at a
// position never change and CTAs do not disturb each other's view of the runs,
// even in place.  Longer runs are left to k_rx_long: a tile in which one of
// them is out of order gets a flag (1: a run from an earlier tile, 2: one that
// starts here and goes on into the next tile, 4: one inside the tile).
// An odd number of passes left the keys in b: every key is then moved to a.
// Measured on 2^28 uniform uint64 keys, in place: 0.64 ms (every
// position tested by its own thread with run scans of its own: 1.0 ms).
constexpr int FN = 256, FL = 64;
template <typename K, int XF>
__global__ void __launch_bounds__(FN) k_rx_fix(RxArgs<K> A)
{
    kernel_entry();
    if (A.nseg > 1 && blockIdx.x >= A.total[2]) return;
    const int64_t seg = A.nseg == 1 ? 0 : A.fix_seg[blockIdx.x];
    const RxPlan& pl = A.plan[seg];
    if (pl.lo == 0) return;
    extern __shared__ __align__(16) char smem[];
    K* sk = (K*)smem;                                 // [FT + 2 * FL + 1]
    uint16_t* runs = (uint16_t*)(sk + FT + 2 * FL + 1);  // [FT / 2 + 1]
    __shared__ unsigned s_runs, s_flag, s_long, s_end;
    __shared__ int s_in;  // first position of the tile after an earlier tile's short run
    int64_t off, len;
    rx_seg(A, seg, off, len);
    const bool move = pl.npass & 1;
    const GBuf<K> dst = rx_global(A.iptr ? rx_own(A.iptr, seg, 0, len) : rx_sub(A.a, off, len));
    const GBuf<K> src = rx_global(move ? rx_sub(A.b, off, len) : dst);
    const typename Rx<K>::M m = Rx<K>::mask(pl.lo, Rx<K>::D - 1);
    const bool inv = !A.keep;
    const int64_t t0 = (int64_t)((int)blockIdx.x - rx_at(A, seg).fix0) * FT, t1 = t0 + FT < len ? t0 + FT : len;
    if (t0 >= len) return;
    const int64_t base = t0 - FL > 0 ? t0 - FL : 0;
    const int end = (int)((t1 + FL + 1 < len ? t1 + FL + 1 : len) - base);  // keys held
    const int h0 = (int)(t0 - base), h1 = (int)(t1 - base);
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_runs = s_flag = s_long = 0;
        s_end = (unsigned)h1;
        s_in = h0;
    }
    constexpr int U = 8;
    for (int i0 = tid; i0 < end; i0 += U * FN) {
        K x[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i0 + u * FN < end) x[u] = src.ld(base + i0 + u * FN);
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i0 + u * FN < end) sk[i0 + u * FN] = inv ? xform<XF>(x[u]) : x[u];
    }
    __syncthreads();
    auto put = [&](int i, const K& x) {
        if (inv) dst.template stx<XF>(base + i, x);
        else dst.st(base + i, x);
    };
#pragma unroll 4
    for (int i = h0 + tid; i < h1; i += FN) {
        const K x = sk[i];
        const bool next = i + 1 < end && Rx<K>::same(sk[i + 1], x, m);
        if (next && !(i > 0 && Rx<K>::same(sk[i - 1], x, m))) runs[atomicAdd(&s_runs, 1u)] = (uint16_t)i;
    }
    if (tid == 0 && h0 > 0 && Rx<K>::same(sk[h0 - 1], sk[h0], m)) {
        // the tile begins inside an earlier tile's run
        const K x = sk[h0];
        int s = h0 - 1;
        while (s > 0 && Rx<K>::same(sk[s - 1], x, m)) s--;
        if (s == 0 || (s + FL < end && Rx<K>::same(sk[s + FL], x, m))) {
            s_long = 1;
        } else {
            int e = h0;
            while (e < end && Rx<K>::same(sk[e], x, m)) e++;
            s_in = e;
        }
    }
    __syncthreads();
    for (unsigned q = tid; q < s_runs; q += FN) {
        const int s = runs[q];
        const K x = sk[s];
        int e = s + 2;
        bool moved = key_lt(sk[s + 1], x);
        while (e < end && e <= s + FL && Rx<K>::same(sk[e], x, m)) {
            moved |= key_lt(sk[e], sk[e - 1]);
            e++;
        }
        if (e > s + FL) {
            s_long = 1;
            continue;
        }
        if (moved) {
            for (int i = s + 1; i < e; i++) {
                const K v = sk[i];
                int j = i;
                for (; j > s && key_lt(v, sk[j - 1]); j--) sk[j] = sk[j - 1];
                sk[j] = v;
            }
            if (!move)
                for (int i = s; i < e; i++) put(i, sk[i]);
        }
        if (e > h1) s_end = (unsigned)e;  // (only the last run reaches beyond the tile)
    }
    __syncthreads();
    if (move) {
        const int i1 = (int)s_end < end ? (int)s_end : end;
        for (int i = s_in + tid; i < i1; i += FN) put(i, sk[i]);
    }
    if (!s_long) return;
    for (int i = h0 + tid; i < h1; i += FN) {
        if (i == 0) continue;
        const K x = sk[i], y = sk[i - 1];
        if (!Rx<K>::same(y, x, m) || !key_lt(x, y)) continue;  // (short runs are in order by now)
        if (i < s_in) continue;
        atomicOr(&s_flag, h0 > 0 && Rx<K>::same(sk[h0 - 1], x, m) ? 1u
                          : h1 < end && Rx<K>::same(sk[h1], x, m) ? 2u
                                                                  : 4u);
    }
    __syncthreads();
    if (tid == 0 && s_flag) {
        A.flags[blockIdx.x] = (uint8_t)s_flag;
        atomicAdd(A.nflag, 1u);
    }
}

// --------------------------------------------------------------- long runs
// Keys of one task of k_rx_long, the longest run that one CTA sorts alone, and CTAs
// per SM.  Tasks of short runs are short, so that all CTAs have some, and those of
// long ones long: each costs some 3 us beside its keys (LONG_T / 2 LONG_T for all runs:
// 2^20 float64 with 30% of the mean 204 / 245 us, 2^24 uint64, half zeros, 831 / 790
// us; 4 LONG_T for 2^30 zeros with rare values below 2^16 16.9 ms, 2 LONG_T 18.4).
constexpr int LONG_T = 8192, LONG_ONE = 2 * LONG_T, LONG_CTAS = 2;
constexpr unsigned LISTED = 128;  // (in RxArgs::flags)
__device__ __forceinline__ int rx_task(int64_t m) { return m < (1 << 22) ? LONG_T : m < (1 << 25) ? 2 * LONG_T : 4 * LONG_T; }
// The first position of [a, b) for which pred fails (it holds for those before),
// by one warp, 32 probes a round.
template <typename F> __device__ __forceinline__ int64_t rx_search(int64_t a, int64_t b, F pred)
{
    const int lane = threadIdx.x & 31;
    while (a < b) {
        const int64_t step = (b - a + 31) / 32, mid = a + (lane + 1) * step - 1;
        const int k = __popc(__ballot_sync(0xFFFFFFFFu, mid < b && pred(mid)));
        const int64_t top = a + (k + 1) * step - 1;
        a += k * step;
        if (a > b) a = b;
        if (top < b) b = top;
    }
    return a;
}
// Lists the runs of the fix tile at t0 that are out of order (one warp; flag: the
// tile's): those inside it as one range, one that goes beyond it once, whichever of
// its tiles comes first.
template <typename K, typename LD>
__device__ __forceinline__ void rx_list(LD ld, int64_t len, int64_t t0, int lo, unsigned flag, int seg, uint8_t* flags,
                                        int64_t fix0, RxBad* bad, unsigned* bads, unsigned maxrows)
{
    const typename Rx<K>::M m = Rx<K>::mask(lo, Rx<K>::D - 1);
    const int64_t t1 = t0 + FT < len ? t0 + FT : len;
    const bool one = (threadIdx.x & 31) == 0;
    auto below = [&](const K& v) { return [&](int64_t i) { return Rx<K>::lt(ld(i), v, m); }; };
    auto upto = [&](const K& v) { return [&](int64_t i) { return !Rx<K>::lt(v, ld(i), m); }; };
    auto list = [&](int64_t s, int64_t e, int inside) {
        if (!one) return;
        const unsigned rows = e - s > LONG_ONE ? (unsigned)((e - s + rx_task(e - s) - 1) / rx_task(e - s)) : 0;
        const unsigned slot = rows ? atomicAdd(bads + 1, rows) : 0u;
        if ((unsigned long long)slot + rows > maxrows) return;  // (only of keys that an abandoned wait left out of order)
        bad[atomicAdd(bads, 1u)] = RxBad{s, e, seg, inside, slot, 0, 0, 0, 0};
    };
    auto spans = [&](int64_t s, int64_t e) {
        const int64_t f = fix0 + s / FT;
        const unsigned bit = LISTED << (8 * (f & 3));
        const unsigned was = one ? atomicOr((unsigned*)(flags + (f & ~int64_t(3))), bit) : 0;
        if ((__shfl_sync(0xFFFFFFFFu, was, 0) & bit) == 0) list(s, e, 0);
    };
    // [in, out): the runs inside the tile
    const K head = ld(t0), tail = ld(t1 - 1);
    const int64_t in = t0 > 0 && Rx<K>::same(ld(t0 - 1), head, m) ? rx_search(t0, t1, upto(head)) : t0;
    if (flag & 1) spans(rx_search(0, t0, below(head)), in < t1 ? in : rx_search(t1, len, upto(head)));
    const int64_t out = t1 < len && Rx<K>::same(ld(t1), tail, m) ? rx_search(in, t1, below(tail)) : t1;
    if ((flag & 2) && out < t1) spans(out, rx_search(t1, len, upto(tail)));
    if (flag & 4) list(in, out, 1);
}
// The bits in which a key differs from another, and the same as a key.
__device__ __forceinline__ void rx_diff(uint64_t x, uint64_t y, unsigned long long& dk, unsigned&) { dk |= x ^ y; }
__device__ __forceinline__ void rx_diff(const Rec& x, const Rec& y, unsigned long long& dk, unsigned& dp)
{
    dk |= x.k ^ y.k;
    dp |= x.p ^ y.p;
}
template <typename K> __device__ __forceinline__ K rx_bits(unsigned long long dk, unsigned) { return dk; }
template <> __device__ __forceinline__ Rec rx_bits<Rec>(unsigned long long dk, unsigned dp) { return Rec{dk, dp}; }
// The bits in which the keys of [a, b) differ from ref, added to *dk and *dp (one
// CTA; in shared or device memory).
template <int NT, typename K, typename LD>
__device__ __forceinline__ void rx_range_bits(LD ld, int64_t a, int64_t b, const K& ref, unsigned long long* dk, unsigned* dp)
{
    unsigned long long vk = 0;
    unsigned vp = 0;
#pragma unroll 8
    for (int64_t i = a + threadIdx.x; i < b; i += NT) rx_diff(ld(i), ref, vk, vp);
    const unsigned lo = __reduce_or_sync(0xFFFFFFFFu, (unsigned)vk), hi = __reduce_or_sync(0xFFFFFFFFu, (unsigned)(vk >> 32));
    vp = __reduce_or_sync(0xFFFFFFFFu, vp);
    if ((threadIdx.x & 31) == 0) {
        if (lo | hi) atomicOr(dk, ((unsigned long long)hi << 32) | lo);
        if (vp) atomicOr(dp, vp);
    }
}
// Whether every thread's digits v[U] are the same in a whole warp.
template <int U> __device__ __forceinline__ bool rx_one_value(const unsigned (&v)[U])
{
    bool same = true;
#pragma unroll
    for (int u = 1; u < U; u++) same &= v[u] == v[0];
    int one;
    __match_all_sync(0xFFFFFFFFu, same ? v[0] : 256u, &one);
    return __all_sync(0xFFFFFFFFu, same) && one;
}
// How often each value of digit d occurs in [a, b), into cnt[256] (one CTA; wt: a
// table per warp).  Long runs mostly hold one value: a warp whose keys all have the
// same digit adds them as one.
template <int NT, typename K, typename LD>
__device__ __forceinline__ void rx_range_count(LD ld, int64_t a, int64_t b, int d, uint32_t* wt, uint32_t* cnt)
{
    constexpr int W = NT / 32, U = 8;
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t* my = wt + (tid >> 5) * 256;
    for (int i = tid; i < W * 256; i += NT) wt[i] = 0;
    __syncthreads();
    for (int64_t c = a; c < b; c += NT * U) {
        unsigned v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = c + u * NT + tid;
            v[u] = Rx<K>::dig(ld(i < b ? i : a), d);
        }
        if (c + NT * U <= b && rx_one_value(v)) {
            if (lane == 0) atomicAdd(&my[v[0]], 32u * U);
            continue;
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (c + u * NT + tid < b) atomicAdd(&my[v[u]], 1u);
    }
    __syncthreads();
    if (tid < 256) {
        uint32_t t = 0;
#pragma unroll
        for (int q = 0; q < W; q++) t += wt[q * 256 + tid];
        cnt[tid] = t;
    }
    __syncthreads();
}
// Exclusive sums over the first 256 threads (red: 8 words of scratch).
__device__ __forceinline__ unsigned long long rx_exsum256(unsigned long long t, unsigned long long* red)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long x = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (w < 8 && lane == 31) red[w] = x;
    __syncthreads();
    x -= t;
    for (int q = 0; q < 8; q++)
        if (q < w) x += red[q];
    __syncthreads();
    return x;
}
// Moves the keys of [a, b) to the places that pos[256] gives for digit d, in order
// (one CTA; keys before `lim` only), and advances pos.
template <int NT, typename K, typename LD, typename ST>
__device__ __forceinline__ void rx_range_scatter(LD ld, ST st, int64_t a, int64_t b, int64_t lim, int d, uint32_t* wt,
                                                 unsigned long long* pos)
{
    constexpr int W = NT / 32, E = 8;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t* my = wt + w * 256;
    for (int64_t c = a; c < b; c += NT * E) {
        const int64_t p0 = c + w * 32 * E + lane;
        for (int i = lane; i < 256; i += 32) my[i] = 0;
        __syncwarp();
        K k[E];
        uint32_t rk[E];
#pragma unroll
        for (int j = 0; j < E; j++) k[j] = ld(p0 + j * 32 < b ? p0 + j * 32 : a);
        unsigned dv[E];
#pragma unroll
        for (int j = 0; j < E; j++) dv[j] = Rx<K>::dig(k[j], d);
        const bool one = c + NT * E <= b && rx_one_value(dv);
        if (one) {
            if (lane == 0) my[dv[0]] = 32 * E;
#pragma unroll
            for (int j = 0; j < E; j++) rk[j] = j * 32 + lane;
        }
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (one) break;
            const bool in = p0 + j * 32 < b;
            const unsigned v = Rx<K>::dig(k[j], d);
            unsigned mt = __ballot_sync(0xFFFFFFFFu, in);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const bool bit = (v >> q) & 1;
                const unsigned u = __ballot_sync(0xFFFFFFFFu, bit);
                mt &= bit ? u : ~u;
            }
            const unsigned r = __popc(mt & ((1u << lane) - 1));
            const uint32_t old = my[v];
            __syncwarp();
            if (in && r == 0) my[v] = old + __popc(mt);
            __syncwarp();
            rk[j] = old + r;
        }
        __syncthreads();
        uint32_t tot = 0;
        if (tid < 256) {
#pragma unroll
            for (int q = 0; q < W; q++) {
                const uint32_t t = wt[q * 256 + tid];
                wt[q * 256 + tid] = tot;
                tot += t;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (p0 + j * 32 >= b) continue;
            const unsigned v = Rx<K>::dig(k[j], d);
            const int64_t p = (int64_t)pos[v] + my[v] + rk[j];
            if (p < lim) st(p, k[j]);
        }
        __syncthreads();
        if (tid < 256) pos[tid] += tot;
    }
    __syncthreads();
}

// Waits until *done reaches `need` (one thread; at most so many looks).
__device__ __forceinline__ bool rx_reached(const unsigned* done, unsigned need, unsigned looks)
{
    for (unsigned spins = 0; spins <= looks; spins++) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
        if (v >= need) return true;
        __nanosleep(100);
    }
    return false;
}

// What k_rx_fix flagged.  All CTAs first list it (a task per LIST fix tiles, taken
// in order from a counter) and wait until the list is whole.  (Listing in k_rx_fix
// cost that kernel 3% where there is nothing to list.)  The runs inside a tile are
// sorted together in shared memory, by one CTA (they lie in order of their leading
// bytes already).  A run that spans tiles is sorted by the bytes left out of the
// passes that vary in it, lowest first, by one CTA alone for up to LONG_ONE keys, by
// all CTAs together for more: its work is cut into tasks, taken in order from a
// counter:
//   differing bits (a task per rx_task keys); then for each varying byte: counts
//   (the same), running sums of them (16), moves (the same); if the moves are odd
//   in number, the way back.
// A task waits until all tasks of the kinds before it are finished; those were
// taken by CTAs that are running, so the waits end whatever share of the grid is
// on the GPU.  So a sample that misjudged the input costs at most the passes it
// saved, each at a grid's full width, and a counting pass each.  A warp whose keys all
// have the same digit, as most of such a run's have, counts and ranks them without
// looking at them one by one; two CTAs per SM hide each other's barriers (one, and every
// key ranked by ballots: 2^30 zeros with rare values below 2^24 50.7 ms, now 25.1).
// Measured, a whole sort (one CTA per run before / this kernel; uniform keys in
// brackets): 2^20 float64 of which 30% are the mean 34.9 / 0.20 ms (0.11), 2^24 uint64
// of which half are zero 1171 / 0.79 ms (0.41), 2^26 int64 zeros with 1e-4 small values
// 7288 / 1.26 ms (1.44), 2^26 records of such keys 8622 / 2.3 ms (2.4).
// Records whose payloads ascend keep that order in a run: equal keys need no
// payload digits.
template <typename K, int XF, typename CT>
__global__ void __launch_bounds__(512, LONG_CTAS) k_rx_long(RxArgs<K> A)
{
    kernel_entry();
    constexpr int NT = 512, E = 8, W = NT / 32;
    static_assert(NT * E == FT, "a fix tile is one shared-memory sort");
    constexpr int LIST = 64;
    if (*A.nflag == 0) return;
    using SB = typename TileBuf<K, E>::type;
    extern __shared__ __align__(16) char smem[];
    uint32_t* wt = (uint32_t*)smem;                              // [W][256]
    unsigned long long* pos = (unsigned long long*)(wt + W * 256);  // [256]
    uint32_t* cnt = (uint32_t*)(pos + 256);                      // [256]
    unsigned long long* red = (unsigned long long*)(cnt + 256);  // [8]
    __shared__ unsigned long long s_dk;
    __shared__ unsigned s_dp, s_t;
    __shared__ bool s_ok;
    const int tid = threadIdx.x;
    const bool inv = !A.keep;
    const bool ascending = sizeof(K) > 8 && *A.descents == 0;
    GBuf<K> x, y;
    int64_t off, len;
    int lo = 0, first = 0;  // the bytes to sort: [first, lo)
    auto open = [&](const RxBad& q) {
        rx_seg(A, (int64_t)q.seg, off, len);
        lo = A.plan[q.seg].lo;
        first = ascending && lo >= 4 ? 4 : 0;
        x = rx_global(A.iptr ? rx_own(A.iptr, (int64_t)q.seg, 0, len) : rx_sub(A.a, off, len));
        y = rx_global(rx_sub(A.b, off, len));
    };
    auto reached = [&](const unsigned* done, unsigned need, unsigned what) {
        if (tid == 0) {
            s_ok = rx_reached(done, need, A.spins);
            if (!s_ok) rx_give_up(A, what);
        }
        __syncthreads();
        const bool ok = s_ok;
        __syncthreads();
        return ok;
    };
    // keys of x, or of y once they are swapped
    auto from = [&](bool swapped) {
        return [&, swapped](int64_t i) {
            const GBuf<K>& b = swapped ? y : x;
            return inv ? b.template ldx<XF>(i) : b.ld(i);
        };
    };
    auto into = [&](bool swapped) {
        return [&, swapped](int64_t i, const K& v) {
            const GBuf<K>& b = swapped ? x : y;
            if (inv) b.template stx<XF>(i, v);
            else b.st(i, v);
        };
    };
    {
        if (A.nseg == 1) rx_seg(A, 0, off, len);  // (its length, not the longest it might have had)
        const int64_t tiles = A.nseg == 1 ? (len + FT - 1) / FT : A.total[2];
        const unsigned tasks = (unsigned)((tiles + LIST - 1) / LIST);
        for (;;) {
            __syncthreads();
            if (tid == 0) s_t = atomicAdd(&A.bads[2], 1u);
            __syncthreads();
            const unsigned t = s_t;
            if (t >= tasks) break;
            const int64_t f0 = (int64_t)t * LIST + (tid >> 5) * (LIST / W);  // a few tiles per warp
            for (int64_t f = f0; f < f0 + LIST / W && f < tiles; f++) {
                const unsigned flag = A.flags[f] & ~LISTED;
                if (flag == 0) continue;
                RxBad q{};
                q.seg = A.nseg == 1 ? 0 : A.fix_seg[f];
                const int fix0 = rx_at(A, q.seg).fix0;
                open(q);
                rx_list<K>(from(false), len, (f - fix0) * FT, lo, flag, q.seg, A.flags, fix0, A.bad, A.bads, A.rows);
            }
            __threadfence();
            __syncthreads();
            if (tid == 0) atomicAdd(&A.bads[3], 1u);
        }
        if (!reached(&A.bads[3], tasks, tasks)) return;
    }
    const unsigned nbad = __ldcg(A.bads);
    for (unsigned r = blockIdx.x; r < nbad; r += gridDim.x) {
        const RxBad q = A.bad[r];
        if (!q.tile && q.e - q.s > LONG_ONE) continue;
        open(q);
        __syncthreads();
        if (q.tile) {
            char* sp = smem;
            const SB sb = SB::carve(sp, FT);
            const int n = (int)(q.e - q.s);
            if (inv) tile_sort_body<NT, E, K, XF, true, 0>(sb, x, q.s, x, q.s, n);
            else tile_sort_body<NT, E, K, 0, true, 0>(sb, x, q.s, x, q.s, n);
            continue;
        }
        if (tid == 0) s_dk = s_dp = 0;
        __syncthreads();
        const auto ld = from(false);
        rx_range_bits<NT, K>(ld, q.s, q.e, ld(q.s), &s_dk, &s_dp);
        __syncthreads();
        const K bits = rx_bits<K>(s_dk, s_dp);
        bool swapped = false;
        for (int d = first; d < lo; d++) {
            if (Rx<K>::dig(bits, d) == 0) continue;
            rx_range_count<NT, K>(from(swapped), q.s, q.e, d, wt, cnt);
            const unsigned long long ex = rx_exsum256(tid < 256 ? cnt[tid] : 0, red);
            if (tid < 256) pos[tid] = (unsigned long long)q.s + ex;
            __syncthreads();
            rx_range_scatter<NT, K>(from(swapped), into(swapped), q.s, q.e, q.e, d, wt, pos);
            swapped = !swapped;
        }
        if (swapped)
            for (int64_t i = q.s + tid; i < q.e; i += NT) x.st(i, y.ld(i));
    }
    // the longest runs, each CTA from a place of its own on, then the others'
    const unsigned start = (unsigned)((unsigned long long)blockIdx.x * nbad / gridDim.x);
    for (unsigned k0 = 0; k0 < nbad; k0 += NT) {
        for (unsigned next = k0;;) {
            __syncthreads();
            if (tid == 0) s_t = ~0u;
            __syncthreads();
            const unsigned k = k0 + tid;
            if (k >= next && k < nbad) {
                const RxBad* q = A.bad + (start + k) % nbad;
                if (!q->tile && q->e - q->s > LONG_ONE) atomicMin(&s_t, k);
            }
            __syncthreads();
            const unsigned pick = s_t;
            if (pick == ~0u) break;
            next = pick + 1;
            RxBad* bad = A.bad + (start + pick) % nbad;
            open(*bad);
            const int64_t s = bad->s, e = bad->e;
            const int T = rx_task(e - s);
            const unsigned nt = (unsigned)((e - s + T - 1) / T);
            CT* table = (CT*)A.dtab + (size_t)bad->slot * 256;  // [256][nt]: counts, then their running sums
            K bits{};
            int digits = -1;  // varying bytes, once known
            for (;;) {
                __syncthreads();
                if (tid == 0) s_t = atomicAdd(&bad->ticket, 1u);
                __syncthreads();
                const unsigned t = s_t;
                if (t < nt) {
                    const auto ld = from(false);
                    const int64_t a = s + (int64_t)t * T, b = a + T < e ? a + T : e;
                    rx_range_bits<NT, K>(ld, a, b, ld(s), &bad->dk, &bad->dp);
                } else {
                    if (digits < 0) {
                        if (!reached(&bad->done, nt, bad->slot)) return;
                        bits = rx_bits<K>(__ldcg(&bad->dk), __ldcg(&bad->dp));
                        digits = 0;
                        for (int d = first; d < lo; d++) digits += Rx<K>::dig(bits, d) != 0;
                    }
                    const unsigned per = 2 * nt + 16;  // tasks of one byte
                    const unsigned di = (t - nt) / per, sub = (t - nt) - di * per;
                    const bool back = (int)di == digits;
                    if ((int)di > digits || (back && (!(digits & 1) || sub >= nt))) break;
                    const unsigned kind = back || sub < nt ? 0 : sub < nt + 16 ? 1 : 2;
                    const unsigned before = nt + di * per + (kind == 0 ? 0 : kind == 1 ? nt : nt + 16);
                    if (!reached(&bad->done, before, bad->slot)) return;
                    int d = first;  // the byte
                    for (unsigned c = 0; d < lo; d++)
                        if (Rx<K>::dig(bits, d) != 0 && c++ == di) break;
                    const bool swapped = di & 1;
                    const unsigned tile = kind == 2 ? sub - nt - 16 : sub;
                    const int64_t a = s + (int64_t)tile * T, b = a + T < e ? a + T : e;
                    if (back) {
                        constexpr int U = 8;
                        for (int64_t i = a + tid; i < b; i += NT * U) {
                            K v[U];
#pragma unroll
                            for (int u = 0; u < U; u++)
                                if (i + u * NT < b) v[u] = y.ld(i + u * NT);
#pragma unroll
                            for (int u = 0; u < U; u++)
                                if (i + u * NT < b) x.st(i + u * NT, v[u]);
                        }
                    } else if (kind == 0) {
                        rx_range_count<NT, K>(from(swapped), a, b, d, wt, cnt);
                        if (tid < 256) table[(size_t)tid * nt + tile] = cnt[tid];
                    } else if (kind == 1) {
                        // a warp per value: inclusive sums of its tiles' counts
                        CT* row = table + (size_t)((sub - nt) * W + (tid >> 5)) * nt;
                        constexpr int U = 8;
                        CT sum = 0;
                        for (unsigned i0 = 0; i0 < nt; i0 += 32 * U) {
                            const unsigned i = i0 + (tid & 31);
                            CT v[U];
#pragma unroll
                            for (int u = 0; u < U; u++) v[u] = i + 32 * u < nt ? __ldcg(row + i + 32 * u) : (CT)0;
#pragma unroll
                            for (int u = 0; u < U; u++) {
#pragma unroll
                                for (int o = 1; o < 32; o <<= 1) {
                                    const CT w = __shfl_up_sync(0xFFFFFFFFu, v[u], o);
                                    if ((tid & 31) >= o) v[u] += w;
                                }
                                v[u] += sum;
                                sum = __shfl_sync(0xFFFFFFFFu, v[u], 31);
                                if (i + 32 * u < nt) row[i + 32 * u] = v[u];
                            }
                        }
                    } else {
                        unsigned long long mine = 0, all = 0;
                        if (tid < 256) {
                            const CT* row = table + (size_t)tid * nt;
                            mine = tile ? (unsigned long long)__ldcg(row + tile - 1) : 0;
                            all = (unsigned long long)__ldcg(row + nt - 1);
                        }
                        const unsigned long long ex = rx_exsum256(all, red);
                        if (tid < 256) pos[tid] = (unsigned long long)s + ex + mine;
                        __syncthreads();
                        rx_range_scatter<NT, K>(from(swapped), into(swapped), a, b, e, d, wt, pos);
                    }
                }
                __threadfence();
                __syncthreads();
                if (tid == 0) atomicAdd(&bad->done, 1u);
            }
        }
    }
}

}  // namespace ps

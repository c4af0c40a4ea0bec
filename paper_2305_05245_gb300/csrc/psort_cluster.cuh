// psort_cluster.cuh -- short sorts in one launch: one thread-block cluster sorts
// a whole instance on chip.
//
// Every CTA of the cluster sorts its share of the keys in its own shared
// memory (tile_sort_body's steps), then log2(cluster size) levels of pairwise
// merges join the shares: at each level a CTA finds by merge path which parts of
// the two runs make up its share of the output, copies them from the other CTAs'
// shared memory (distributed shared memory) into its own and merges them there.
// The keys are read from and written to device memory once, and no workspace is
// needed.
#pragma once

#include "psort_kernels.cuh"

namespace ps {

__device__ __forceinline__ unsigned cl_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Barrier over all threads of the cluster; shared-memory writes before it are
// seen by every CTA after it.
__device__ __forceinline__ void cl_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The same shared-memory address in the CTA of the given rank.
template <typename P> __device__ __forceinline__ P* cl_map(P* p, unsigned rank)
{
    P* q;
    asm("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
    return q;
}
template <typename K, int W> __device__ __forceinline__ SBuf<K, W> cl_buf(const SBuf<K, W>& b, unsigned rank)
{
    return SBuf<K, W>{cl_map(b.a, rank), b.cap};
}
template <int W> __device__ __forceinline__ SBuf<Rec, W> cl_buf(const SBuf<Rec, W>& b, unsigned rank)
{
    SBuf<Rec, W> q;
    q.k = cl_buf(b.k, rank);
    q.p = cl_buf(b.p, rank);
    return q;
}

// Sorts block blockIdx.x / CS of the instances' n_B blocks each; share: keys per
// CTA, a multiple of E, at most NT*E, with CS * share no less than the longest
// block.  src and dst may be the same buffer (every key is read before the first
// barrier and written after the last).  iptr (keys only, n_B = 1): instances in
// buffers of their own.  keep: the result stays order keys.
//
// Latency bound: one cluster, a CTA of up to 32 warps per SM.  Shares of 1024 x 4
// keys take half the merge work per thread of 1024 x 8 and are used while they
// fit.  Measured per call, a tile sort, planning kernels and a chunk merge before
// / this kernel: 2^15 int32 85 / 31 us, 2^16 89 / 40 us, 40961 int64 (with a copy of
// the keys) 84.7 / 34.8 us.
template <int NT, int E, typename K, int XF, int WLEV, int CS>
__global__ void __launch_bounds__(NT, 1) k_cluster_sort(GBuf<K> src, GBuf<K> dst, Inst in, int64_t n_B, int share, K* const* iptr, bool keep)
{
    kernel_entry();
    constexpr int T = NT * E;
    using SB = typename TileBuf<K, E>::type;
    using SV = typename ViewOf<SB>::type;
    extern __shared__ __align__(16) char smem[];
    char* sp = smem;
    const SB sb = SB::carve(sp, T);
    const int64_t inst = n_B == 1 ? blockIdx.x / CS : blockIdx.x / CS / n_B;
    const unsigned c = CS > 1 ? cl_rank() : 0;
    int64_t bs = 0, be = in.len(inst);
    if (n_B > 1) block_bounds(in.len(inst), n_B, blockIdx.x / CS - inst * n_B, bs, be);
    const int64_t N = be - bs;
    const int64_t o = in.off(inst) + bs + (int64_t)c * share;
    const int64_t left = N - (int64_t)c * share;
    const int n = left <= 0 ? 0 : (int)(left < share ? left : share);  // this CTA's keys
    const int tid = threadIdx.x;
    {
        K r[E];
        if constexpr (sizeof(K) <= 8) {
            if (iptr) tile_load_regs<NT, E, K, XF>(GBuf<K>{iptr[inst], N}, (int64_t)c * share, n, r);
            else tile_load_regs<NT, E, K, XF>(src, o, n, r);
        } else {
            tile_load_regs<NT, E, K, XF>(src, o, n, r);
        }
        reg_sort<E>(r);
        if constexpr (WLEV > 0) warp_merge_levels<E, WLEV>(r);
        store_bitonic<E>(SV{sb}, tid * E, E << WLEV, (E << WLEV) >= T, r);
    }
    __syncthreads();
    merge_levels_pow2<NT, E>(SV{sb}, E << (WLEV + 1));
    if constexpr (CS > 1) {
        // the first `share` keys of every CTA's buffer now are a sorted run
        // (missing keys count as the largest key)
        const SB tb = SB::carve(sp, T);
        __shared__ int s_a[2];
        const int lane = tid & 31, w = tid >> 5;
        const unsigned inv = (unsigned)((0x100000000ull + share - 1) / share);  // i / share = mulhi(i, inv) below 2^17
        cl_sync();
#pragma unroll 1
        for (int half = 1; half < CS; half *= 2) {
            const unsigned u = c & ~(2u * half - 1);  // first CTA of the pair of runs
            const int run = half * share;
            auto at = [&](unsigned first, int i) {
                const unsigned q = __umulhi((unsigned)i, inv);
                return cl_buf(sb, first + q).ld(i - (int)q * share);
            };
            const int d0 = (int)(c - u) * share;
            if (w < 2) {
                // co-rank of output d (warp 0: the share's first, warp 1: its end):
                // the elements of the lower run among the first d outputs, by 32
                // probes a round
                const int d = d0 + w * share;
                int lo = d > run ? d - run : 0, hi = d < run ? d : run;
                while (lo < hi) {
                    const int step = (hi - lo + 31) / 32, mid = lo + lane * step;
                    const bool p = mid < hi && !SV::lt(at(u + half, d - 1 - mid), at(u, mid));
                    const int k = __popc(__ballot_sync(0xFFFFFFFFu, p));
                    if (k == 0) break;
                    const int top = lo + k * step;
                    lo += (k - 1) * step + 1;
                    if (top < hi) hi = top;
                }
                if (lane == 0) s_a[w] = lo;
            }
            __syncthreads();
            const int a0 = s_a[0], la = s_a[1] - a0, b0 = d0 - a0;
            {
                K x[E];
#pragma unroll
                for (int j = 0; j < E; j++) {
                    const int i = tid + j * NT;
                    if (i < share) x[j] = i < la ? at(u, a0 + i) : at(u + half, b0 + i - la);
                }
#pragma unroll
                for (int j = 0; j < E; j++)
                    if (tid + j * NT < share) tb.st(tid + j * NT, x[j]);
            }
            cl_sync();  // every CTA has its copies: the runs may be overwritten
            const int pos0 = tid * E;
            if (pos0 < share) {
                K out[E];
                const int x = merge_path(SV{tb}, 0, la, share, pos0);
                serial_merge<E, false>(SV{tb}, x, la, la + pos0 - x, share, E, out);
                store_block<E>(SV{sb}, pos0, out);
            }
            if (2 * half < CS) cl_sync();
            else __syncthreads();
        }
    }
    if constexpr (sizeof(K) <= 8) {
        if (iptr) {
            const GBuf<K> own{iptr[inst], N};
            for (int i = tid; i < n; i += NT) own.template stx<XF>((int64_t)c * share + i, sb.ld(i));
            return;
        }
    }
    if (keep)
        for (int i = tid; i < n; i += NT) dst.st(o + i, sb.ld(i));
    else
        for (int i = tid; i < n; i += NT) dst.template stx<XF>(o + i, sb.ld(i));
}

}  // namespace ps

// psort_struct.cu -- sorting fixed-size records by an embedded uint64 key
// (Table 1's Pair and Particle inputs).  The four steps run on (key,
// position) pairs; the records themselves move once, by a gather.
#include "psort_internal.h"

namespace ps {

// The split moves records in words of 16 or 8 bytes (W), a batch of `per` records
// (up to BATCH words) per CTA and round; consecutive threads take consecutive words,
// four loads in flight each.  The record of a word comes from one multiply (j *
// words < 2^32 for j < BATCH + 1024).  Bound by device memory: 10^7 records of 96
// bytes (1.9 GB) 455 -> 325 us (a 64-bit division per word and one load in flight
// before).  The same for the gather changed nothing (440 us): its reads go to random
// places.
constexpr int BATCH = 4096, UNROLL = 4, NT = 256;

__device__ __forceinline__ uint64_t half_of(const uint4& v, int h)
{
    return h ? ((uint64_t)v.w << 32) | v.z : ((uint64_t)v.y << 32) | v.x;
}
__device__ __forceinline__ uint64_t half_of(const uint64_t& v, int) { return v; }

// Copy every record into the workspace and pull out its key and position: word
// key_word of record i holds (in its half key_half) keys[i]; pos[i] = i.
template <typename W>
__global__ void __launch_bounds__(NT) k_struct_split(const W* rec, W* copy, int64_t n, int words, int per,
                                                     int key_word, int key_half, uint64_t* keys, uint32_t* pos)
{
    const unsigned inv = (unsigned)((0x100000000ull + words - 1) / words);
    for (int64_t r0 = (int64_t)blockIdx.x * per; r0 < n; r0 += (int64_t)gridDim.x * per) {
        const int cnt = (int)(n - r0 < per ? n - r0 : per) * words;
        const W* src = rec + r0 * words;
        W* dst = copy + r0 * words;
        for (int j0 = threadIdx.x; j0 < cnt; j0 += NT * UNROLL) {
            W v[UNROLL];
#pragma unroll
            for (int u = 0; u < UNROLL; u++)
                if (j0 + u * NT < cnt) v[u] = src[j0 + u * NT];
#pragma unroll
            for (int u = 0; u < UNROLL; u++) {
                const int j = j0 + u * NT;
                if (j >= cnt) continue;
                dst[j] = v[u];
                const int r = words == 1 ? j : (int)__umulhi((unsigned)j, inv);
                if (j - r * words == key_word) {
                    keys[r0 + r] = half_of(v[u], key_half);
                    pos[r0 + r] = (uint32_t)(r0 + r);
                }
            }
        }
    }
}

// records[i] = copy[pos[i]], W-sized words (8 or 16 bytes), one thread per
// word of the output (coalesced stores; each record is read contiguously).  A
// position is below n unless the sort before lost keys (a wait that gave up).
template <typename W>
__global__ void k_struct_gather(const W* copy, W* rec, const uint32_t* pos, int64_t words_total, int words, uint32_t n)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < words_total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / words;
        const int w = (int)(t - i * words);
        const uint32_t at = pos[i];
        rec[t] = copy[(int64_t)(at < n ? at : 0) * words + w];
    }
}

static unsigned grid_for(int64_t work)
{
    const int64_t g = (work + 255) / 256;
    return (unsigned)std::min<int64_t>(g, 152 * 16);
}

int struct_sort(void* records, int64_t n, int64_t rb, int64_t ko, int mode, const ps_params* params,
                cudaStream_t s)
{
    const size_t copy_bytes = (size_t)n * (size_t)rb;
    const size_t pair_off = (copy_bytes + 255) & ~(size_t)255;
    const size_t pos_off = pair_off + (((size_t)n * 8 + 255) & ~(size_t)255);
    const size_t total = pos_off + (size_t)n * 4;
    char* ws = nullptr;
    int rc = ws_alloc((void**)&ws, total, s);
    if (rc != PS_OK) return rc;
    uint64_t* keys = (uint64_t*)(ws + pair_off);
    uint32_t* pos = (uint32_t*)(ws + pos_off);
    const bool wide = rb % 16 == 0 && (uintptr_t)records % 16 == 0;
    const int words = (int)(rb / (wide ? 16 : 8));
    // records per batch: at most BATCH words, enough batches to fill the GPU, a word per thread
    const int per = (int)std::max<int64_t>((NT + words - 1) / words, std::min<int64_t>(BATCH / words, n / (152 * 8)));
    const unsigned grid = (unsigned)std::min<int64_t>((n + per - 1) / per, 152 * 16);
    const int64_t wt = n * words;
    {
        ProfScope ps_("struct_split", s);
        if (wide)
            k_struct_split<uint4><<<grid, NT, 0, s>>>((const uint4*)records, (uint4*)ws, n, words, per, (int)(ko / 16),
                                                      (int)(ko / 8 % 2), keys, pos);
        else
            k_struct_split<uint64_t><<<grid, NT, 0, s>>>((const uint64_t*)records, (uint64_t*)ws, n, words, per,
                                                         (int)(ko / 8), 0, keys, pos);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        rc = sort_records(keys, pos, n, mode, params, s);
        if (rc == PS_OK) {
            ProfScope ps_("struct_gather", s);
            if (wide)
                k_struct_gather<uint4><<<grid_for(wt), 256, 0, s>>>((const uint4*)ws, (uint4*)records, pos, wt, words, (uint32_t)n);
            else
                k_struct_gather<uint64_t><<<grid_for(wt), 256, 0, s>>>((const uint64_t*)ws, (uint64_t*)records, pos, wt, words, (uint32_t)n);
            e = cudaGetLastError();
        }
    }
    ws_free(ws, s);
    if (rc != PS_OK) return rc;
    if (e != cudaSuccess) return fail_cuda(e);
    return PS_OK;
}

}  // namespace ps

// psort_cluster_run.cuh -- host side of the one-launch sorts: shape by size.
#pragma once

#include "psort_cluster.cuh"
#include "psort_pipeline.cuh"

namespace ps {

template <typename K> struct ClusterSort {
    static constexpr int TW = Cfg<K>::TW;  // warp-shuffle levels of the tile sort

    struct Job {
        GBuf<K> src, dst;
        Inst in;
        int64_t n_B;  // blocks per instance
        K* const* own;
        bool keep;
        cudaStream_t stream;
    };
    template <int NT, int E, int XF, int CS> static cudaError_t launch(const Job& j, int64_t nmax)
    {
        using SB = typename TileBuf<K, E>::type;
        auto f = k_cluster_sort<NT, E, K, XF, TW, CS>;
        const size_t sm = SB::bytes(NT * E) * (CS > 1 ? 2 : 1) + 64;
        cudaError_t e = smem_attr(f, sm, CS > 8);
        if (e != cudaSuccess) return e;
        const int share = (int)(((nmax + CS - 1) / CS + E - 1) / E * E);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(j.in.count * j.n_B * CS));
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = sm;
        cfg.stream = j.stream;
        cudaLaunchAttribute at[2] = {};
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // (see launch_next)
        at[0].val.programmaticStreamSerializationAllowed = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim.x = CS;
        at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = CS > 1 ? 2 : 1;
        ProfScope ps_("cluster_sort", j.stream);
        return cudaLaunchKernelEx(&cfg, f, j.src, j.dst, j.in, j.n_B, share, j.own, j.keep);
    }

    // Whether a cluster of so many CTAs of the widest shape fits the current device.
    static bool placeable(int ctas)
    {
        using SB = typename TileBuf<K, 8>::type;
        auto f = k_cluster_sort<1024, 8, K, 0, TW, 16>;
        const size_t sm = SB::bytes(8192) * 2 + 64;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3(1024);
        cfg.dynamicSmemBytes = sm;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)ctas;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        if (smem_attr(f, sm, true) == cudaSuccess && cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess) return n > 0;
        cudaGetLastError();
        return false;
    }

    // Small shapes first: one CTA while a tile holds the keys, then clusters of 4
    // and 16 (more, shorter shares sort sooner: 16384 keys in 4 x 4096, not 2 x 8192).
    template <int XF> static cudaError_t run_xf(const Job& j, int64_t n)
    {
        if (n <= 1024) return launch<128, 8, XF, 1>(j, n);
        if (n <= 2048) return launch<256, 8, XF, 1>(j, n);
        if (n <= 4096) return launch<1024, 4, XF, 1>(j, n);
        if (n <= 8192) return launch<1024, 8, XF, 1>(j, n);
        if (n <= 16384) return launch<1024, 4, XF, 4>(j, n);
        if (n <= 65536) return launch<1024, 4, XF, 16>(j, n);
        return launch<1024, 8, XF, 16>(j, n);
    }

    // Many blocks (step 1 of a sort whose blocks were given): the fewest CTAs each.
    template <int XF> static cudaError_t blocks_xf(const Job& j, int64_t L)
    {
        if (L <= 4096) return launch<1024, 4, XF, 1>(j, L);
        if (L <= 8192) return launch<1024, 8, XF, 1>(j, L);
        if (L <= 16384) return launch<1024, 8, XF, 2>(j, L);
        if (L <= 32768) return launch<1024, 8, XF, 4>(j, L);
        if (L <= 65536) return launch<1024, 8, XF, 8>(j, L);
        return launch<1024, 8, XF, 16>(j, L);
    }
    static cudaError_t blocks(int xf, const GBuf<K>& src, const GBuf<K>& dst, const Inst& in, int64_t n_B, int64_t L,
                              cudaStream_t s)
    {
        const Job j{src, dst, in, n_B, nullptr, true, s};
        if constexpr (sizeof(K) > 8) return blocks_xf<0>(j, L);
        else return xf == 1 ? blocks_xf<1>(j, L) : xf == 2 ? blocks_xf<2>(j, L) : blocks_xf<0>(j, L);
    }

    // One launch sorts every instance of a (at most CLUSTER_MAX keys each).
    static int run(const SortArgs& a)
    {
        Inst in;
        in.base = a.inst_base;
        in.n = a.inst_n;
        in.count = a.n_inst;
        in.n0 = a.n;
        const int64_t n = a.inst_base ? a.n_max : a.n;
        if (n > CLUSTER_MAX) return PS_ERR_INVALID_ARG;
        const GBuf<K> user = gbuf_user<K>(a);
        Job j{gbuf_ext<K>(a.src_keys, user), gbuf_ext<K>(a.dst_keys, user), in, 1, nullptr, false, a.stream};
        if constexpr (sizeof(K) <= 8) j.own = (K* const*)a.inst_ptrs;
        cudaError_t e;
        if constexpr (sizeof(K) > 8) {
            e = run_xf<0>(j, n);
        } else {
            switch (xf_of(a.dtype)) {
            case 1: e = run_xf<1>(j, n); break;
            case 2: e = run_xf<2>(j, n); break;
            default: e = run_xf<0>(j, n); break;
            }
        }
        return e == cudaSuccess ? PS_OK : fail_cuda(e);
    }
};

}  // namespace ps

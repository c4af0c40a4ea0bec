// psort_radix_run.cuh -- host side of the radix block sort: workspace layout
// and launches.
#pragma once

#include "psort_internal.h"
#include "psort_pipeline.cuh"
#include "psort_radix.cuh"

namespace ps {

// Threads, keys per thread and CTAs per SM of a digit pass.
template <typename K> struct RxCfg;
template <> struct RxCfg<uint32_t> { static constexpr int NT = 512, E = 24, CTAS = 2; };
template <> struct RxCfg<uint64_t> { static constexpr int NT = 512, E = 16, CTAS = 2; };

template <typename K> struct Radix {
    using C = RxCfg<K>;
    static constexpr int D = Rx<K>::D, T = C::NT * C::E;
    static constexpr int G = 4, CNT = 512;  // digits and threads of a counting CTA

    struct Layout {
        int64_t nseg, R, ntiles, chunk, RC;
        bool wide;  // 64-bit look-back words
        size_t o_hist, o_done, o_ticket, o_lb0, zero_bytes, o_lb1, o_plan, o_data, total;
    };
    static Layout layout(const SortArgs& a)
    {
        Layout y;
        const int64_t nmax = a.inst_base ? a.n_max : a.n, extent = a.inst_base ? a.extent : a.n;
        y.nseg = a.n_inst;
        y.R = (nmax + T - 1) / T;
        y.ntiles = y.nseg * y.R;
        y.wide = nmax >= (int64_t(1) << 30);
        // counting chunks: about four per SM, 4096 to 2^20 keys
        const int64_t want = (nmax * y.nseg) / (152 * 4);
        y.chunk = std::min<int64_t>(int64_t(1) << 20, std::max<int64_t>(4096, (want + 4095) / 4096 * 4096));
        y.RC = (nmax + y.chunk - 1) / y.chunk;
        const size_t lb = align256((size_t)y.ntiles * 256 * (y.wide ? 8 : 4));
        size_t o = 0;
        y.o_hist = o;
        o += align256((size_t)y.nseg * D * 256 * 8);
        y.o_done = o;
        o += align256((size_t)y.nseg * 4);
        y.o_ticket = o;
        o += 256;
        y.o_lb0 = o;
        o += lb;
        y.zero_bytes = o;  // everything up to here starts as zeros
        y.o_lb1 = o;
        o += lb;
        y.o_plan = o;
        o += align256((size_t)y.nseg * sizeof(RxPlan));
        y.o_data = o;
        o += align256((size_t)extent * GStore<K>::bytes + 256);
        y.total = o;
        return y;
    }

    template <int XF, typename CT>
    static cudaError_t passes(const SortArgs& a, const Layout& y, const RxArgs<K>& A, char* ws, int grid_sms)
    {
        cudaStream_t s = a.stream;
        auto fc = k_rx_count<CNT, G, K, XF>;
        const size_t cb = (size_t)G * 4096 * 4;
        cudaError_t e = smem_attr(fc, cb);
        if (e != cudaSuccess) return e;
        {
            ProfScope ps_("radix_count", s);
            fc<<<dim3((unsigned)(y.nseg * y.RC), D / G), CNT, cb, s>>>(A);
        }
        auto fp = k_rx_pass<K, XF, CT, C::NT, C::E, C::CTAS>;
        constexpr size_t sb = rx_smem<K, CT, C::NT, C::E>();
        if ((e = smem_attr(fp, sb)) != cudaSuccess) return e;
        const unsigned grid = (unsigned)std::min<int64_t>(y.ntiles, (int64_t)grid_sms * C::CTAS);
        CT* l0 = (CT*)(ws + y.o_lb0);
        CT* l1 = (CT*)(ws + y.o_lb1);
        for (int i = 0; i < D; i++) {
            ProfScope ps_("radix_pass", s);
            fp<<<grid, C::NT, sb, s>>>(A, i, (i & 1) ? l1 : l0, (i & 1) ? l0 : l1);
        }
        return cudaGetLastError();
    }

    template <int XF> static cudaError_t run_xf(const SortArgs& a, const Layout& y, char* ws)
    {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, y.zero_bytes, a.stream);
        if (e != cudaSuccess) return e;
        RxArgs<K> A;
        A.a = gbuf_user<K>(a);
        A.b = gbuf_at<K>(ws + y.o_data, a.inst_base ? a.extent : a.n);
        A.first = gbuf_ext<K>(a.src_keys, A.a);
        A.last = gbuf_ext<K>(a.dst_keys, A.a);
        A.in.base = a.inst_base;
        A.in.n = a.inst_n;
        A.in.count = a.n_inst;
        A.in.n0 = a.n;
        A.n_B = 1;
        A.nseg = y.nseg;
        A.R = y.R;
        A.ntiles = y.ntiles;
        A.iptr = (K* const*)a.inst_ptrs;
        A.hist = (unsigned long long*)(ws + y.o_hist);
        A.plan = (RxPlan*)(ws + y.o_plan);
        A.done = (unsigned*)(ws + y.o_done);
        A.ticket = (unsigned*)(ws + y.o_ticket);
        A.chunk = y.chunk;
        A.RC = y.RC;
        A.keep = a.keep_order_keys;
        // a sort between two buffers, or one that leaves order keys, moves
        // (and transforms) the keys even when they are all equal
        A.min_pass = (A.keep || a.src_keys || a.dst_keys) ? 2 : 0;
        return y.wide ? passes<XF, uint64_t>(a, y, A, ws, sms) : passes<XF, uint32_t>(a, y, A, ws, sms);
    }

    static int run(const SortArgs& a)
    {
        const Layout y = layout(a);
        char* ws = nullptr;
        const int rc = ws_alloc((void**)&ws, y.total, a.stream);
        if (rc != PS_OK) return rc;
        cudaError_t e;
        switch (xf_of(a.dtype)) {
        case 1: e = run_xf<1>(a, y, ws); break;
        case 2: e = run_xf<2>(a, y, ws); break;
        default: e = run_xf<0>(a, y, ws); break;
        }
        ws_free(ws, a.stream);
        return e == cudaSuccess ? PS_OK : fail_cuda(e);
    }
};

// The first abandoned look-back wait (site 90, index = tile) or, in checked
// builds, the first index violation of this translation unit's kernels; clears
// the record.  Returns 1 if there was one, 0 if none.
static int rx_viol_read(unsigned long long* out)
{
    unsigned long long stall = 0;
    const unsigned long long zero[4] = {0, 0, 0, 0};
    for (int i = 0; i < 4; i++) out[i] = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&stall, rx_stall, sizeof(stall));
    if (e == cudaSuccess && stall) {
        out[0] = 90;
        out[1] = stall - 1;
        e = cudaMemcpyToSymbol(rx_stall, zero, sizeof(stall));
    }
#ifdef PS_CHECKED
    if (e == cudaSuccess && !out[0]) {
        e = cudaMemcpyFromSymbol(out, ps_viol, sizeof(zero));
        if (e == cudaSuccess) e = cudaMemcpyToSymbol(ps_viol, zero, sizeof(zero));
    }
#endif
    if (e != cudaSuccess) return fail_cuda(e);
    return out[0] ? 1 : 0;
}

}  // namespace ps

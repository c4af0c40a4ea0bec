// psort_radix_run.cuh -- host side of the radix block sort: workspace layout
// and launches.
#pragma once

#include "psort_internal.h"
#include "psort_pipeline.cuh"
#include "psort_radix.cuh"

namespace ps {

// Threads, keys per thread and CTAs per SM of a digit pass.  Large tiles spread
// the fixed work of a tile (digit tables, look-back, barriers) over more keys;
// sorts of few tiles want more of them at once.  Measured per sort: uint32,
// 512 x 24 / 384 x 32 / 256 x 32 / 512 x 16: 2^28 keys 3.48 / 3.50 / 3.53 / 4.00
// ms, 2^22 129 / 135 / 141 / 124 us, and 512 x 8 against 512 x 16 at 2^18 62 / 71
// us; uint64, 384 x 24 / 256 x 32 / 512 x 16: 2^28 5.54 / 5.58 / 5.64 ms; records,
// 384 x 16 / 256 x 24 / 512 x 12: 2^28 8.90 / 9.00 / 9.05 ms.
template <int NT_, int E_, int CTAS_> struct RxShape {
    static constexpr int NT = NT_, E = E_, CTAS = CTAS_, T = NT_ * E_;
};
template <typename K> struct RxCfg;
template <> struct RxCfg<uint32_t> {
    using Small = RxShape<512, 8, 2>;
    using Mid = RxShape<512, 16, 2>;
    using Large = RxShape<512, 24, 2>;
    static constexpr int64_t small = int64_t(1) << 18, mid = int64_t(1) << 23;  // up to so many keys
};
template <> struct RxCfg<uint64_t> {
    using Small = RxShape<512, 8, 2>;
    using Mid = RxShape<384, 24, 2>;
    using Large = RxShape<384, 24, 2>;
    static constexpr int64_t small = int64_t(1) << 18, mid = int64_t(1) << 18;
};
template <> struct RxCfg<Rec> {
    using Small = RxShape<512, 8, 2>;
    using Mid = RxShape<384, 16, 2>;
    using Large = RxShape<384, 16, 2>;
    static constexpr int64_t small = int64_t(1) << 18, mid = int64_t(1) << 18;
};

template <typename K> struct Radix {
    using C = RxCfg<K>;
    static constexpr int D = Rx<K>::D;
    static constexpr int G = 4, CNT = 512;  // digits and threads of a counting CTA

    struct Layout {
        int T;  // keys per tile
        int64_t nseg, R, ntiles, chunk, RC;
        bool wide;  // 64-bit look-back words
        int S;      // sampled keys (0: every digit is sorted)
        size_t o_nflag, o_hits, o_tab, o_flags;
        size_t o_hist, o_done, o_ticket, o_lb0, zero_bytes, o_lb1, o_plan, o_data, total;
    };
    static Layout layout(const SortArgs& a)
    {
        Layout y;
        const int64_t nmax = a.inst_base ? a.n_max : a.n, extent = a.inst_base ? a.extent : a.n;
        y.nseg = a.n_inst;
        y.T = nmax <= C::small ? C::Small::T : nmax <= C::mid ? C::Mid::T : C::Large::T;
        y.R = (nmax + y.T - 1) / y.T;
        y.ntiles = y.nseg * y.R;
        y.wide = nmax >= (int64_t(1) << 30);
        // counting chunks: about four per SM, 4096 to 2^20 keys
        const int64_t want = (nmax * y.nseg) / (152 * 4);
        y.chunk = std::min<int64_t>(int64_t(1) << 20, std::max<int64_t>(4096, (want + 4095) / 4096 * 4096));
        y.RC = (nmax + y.chunk - 1) / y.chunk;
        // sqrt(8 n) sampled keys: runs of about one key out of order then give
        // two hits, the least that tells them from none
        y.S = 0;
        if (D > 4 && y.nseg == 1) {
            y.S = 256;
            while (y.S < RX_SAMPLE_MAX && (int64_t)y.S * y.S < 8 * nmax) y.S *= 2;
        }
        const size_t lb = align256((size_t)y.ntiles * 256 * (y.wide ? 8 : 4));
        size_t o = 0;
        y.o_hist = o;
        o += align256((size_t)y.nseg * D * 256 * 8);
        y.o_done = o;
        o += align256((size_t)y.nseg * 4);
        y.o_ticket = o;
        o += 256;
        y.o_nflag = o;
        y.o_hits = o + 8;
        o += 256;
        y.o_tab = o;
        o += align256((size_t)(y.S ? D : 0) * 2 * y.S * 4);
        y.o_flags = o;
        o += align256(y.S ? (size_t)(nmax + FT - 1) / FT : 0);
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

    template <int XF, typename CT, typename SH>
    static cudaError_t digits(const Layout& y, const RxArgs<K>& A, char* ws, int grid_sms, cudaStream_t s)
    {
        auto fp = k_rx_pass<K, XF, CT, SH::NT, SH::E, SH::CTAS>;
        constexpr size_t sb = rx_smem<K, CT, SH::NT, SH::E>();
        cudaError_t e = smem_attr(fp, sb);
        if (e != cudaSuccess) return e;
        const unsigned grid = (unsigned)std::min<int64_t>(y.ntiles, (int64_t)grid_sms * SH::CTAS);
        CT* l0 = (CT*)(ws + y.o_lb0);
        CT* l1 = (CT*)(ws + y.o_lb1);
        for (int i = 0; i < D; i++) {
            ProfScope ps_("radix_pass", s);
            fp<<<grid, SH::NT, sb, s>>>(A, i, (i & 1) ? l1 : l0, (i & 1) ? l0 : l1);
        }
        return cudaGetLastError();
    }

    template <int XF, typename CT>
    static cudaError_t passes(const SortArgs& a, const Layout& y, const RxArgs<K>& A, char* ws, int grid_sms)
    {
        cudaStream_t s = a.stream;
        cudaError_t e;
        if constexpr (D > 4) {
            if (y.S) {
                ProfScope ps_("radix_sample", s);
                k_rx_sample<K, XF><<<dim3((unsigned)((y.S + 127) / 128), D - 2), 128, 0, s>>>(
                    A, (unsigned*)(ws + y.o_tab));
            }
        }
        auto fc = k_rx_count<CNT, G, K, XF>;
        const size_t cb = (size_t)G * 4096 * 4;
        if ((e = smem_attr(fc, cb)) != cudaSuccess) return e;
        {
            ProfScope ps_("radix_count", s);
            fc<<<dim3((unsigned)(y.nseg * y.RC), D / G), CNT, cb, s>>>(A);
        }
        if (std::is_same<CT, uint32_t>::value && y.T == C::Small::T)
            e = digits<XF, uint32_t, typename C::Small>(y, A, ws, grid_sms, s);
        else if (std::is_same<CT, uint32_t>::value && y.T == C::Mid::T)
            e = digits<XF, uint32_t, typename C::Mid>(y, A, ws, grid_sms, s);
        else
            e = digits<XF, CT, typename C::Large>(y, A, ws, grid_sms, s);
        if (e != cudaSuccess) return e;
        if constexpr (D > 4) {
            if (y.S) {
                {
                    auto ff = k_rx_fix<K, XF>;
                    constexpr size_t fb = sizeof(K) * (FT + 2 * FL + 1) + 2 * (FT / 2 + 2);
                    if ((e = smem_attr(ff, fb)) != cudaSuccess) return e;
                    ProfScope ps_("radix_fix", s);
                    ff<<<(unsigned)((A.in.n0 + FT - 1) / FT), FN, fb, s>>>(A);
                }
                ProfScope ps_("radix_long", s);
                k_rx_long<K, XF><<<(unsigned)grid_sms, 512, 0, s>>>(A);
            }
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
        A.iptr = std::is_same<K, Rec>::value ? nullptr : (K* const*)a.inst_ptrs;
        A.hist = (unsigned long long*)(ws + y.o_hist);
        A.plan = (RxPlan*)(ws + y.o_plan);
        A.done = (unsigned*)(ws + y.o_done);
        A.ticket = (unsigned*)(ws + y.o_ticket);
        A.chunk = y.chunk;
        A.RC = y.RC;
        A.sample = y.S;
        A.hits = (unsigned*)(ws + y.o_hits);
        A.nflag = (unsigned*)(ws + y.o_nflag);
        A.flags = (uint8_t*)(ws + y.o_flags);
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
        if constexpr (std::is_same<K, Rec>::value) {
            e = run_xf<0>(a, y, ws);
        } else {
            switch (xf_of(a.dtype)) {
            case 1: e = run_xf<1>(a, y, ws); break;
            case 2: e = run_xf<2>(a, y, ws); break;
            default: e = run_xf<0>(a, y, ws); break;
            }
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

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
        int64_t nseg, tiles, chunk, chunks, fixes, S;  // (several segments: upper bounds)
        bool wide;     // 64-bit look-back words
        size_t o_hist, o_done, o_ticket, o_misc, o_hits, o_tab, o_flags, o_lb0, zero_bytes, o_lb1, o_plan, o_at, o_tile,
            o_chunk, o_fix, o_data, total;
    };
    static Layout layout(const SortArgs& a)
    {
        Layout y;
        const bool multi = a.inst_base != nullptr;
        const int64_t nmax = multi ? a.n_max : a.n, nsum = multi ? a.n_sum : a.n, extent = multi ? a.extent : a.n;
        y.nseg = a.n_inst;
        const int64_t extra = y.nseg == 1 ? 0 : y.nseg;
        auto parts = [&](int64_t u) { return y.nseg == 1 ? (nsum + u - 1) / u : nsum / u + extra; };
        y.T = nsum <= C::small ? C::Small::T : nsum <= C::mid ? C::Mid::T : C::Large::T;
        y.tiles = parts(y.T);
        y.wide = nmax >= (int64_t(1) << 30);
        // counting chunks: about four per SM, 4096 to 2^20 keys (2^16 for several segments)
        const int64_t want = nsum / (152 * 4);
        y.chunk = std::min<int64_t>(int64_t(1) << (extra ? 16 : 20), std::max<int64_t>(4096, (want + 4095) / 4096 * 4096));
        y.chunks = parts(y.chunk);
        const bool sampled = D > 4;
        y.fixes = sampled ? parts(FT) : 0;
        y.S = sampled ? rx_samples(nmax) : 0;
        // hash tables: S < 2 sqrt(8 n), or 128, keys of each segment
        const double many = y.nseg == 1 ? (double)y.S : 2.0 * std::sqrt(8.0 * (double)y.nseg * (double)nsum) + 128.0 * y.nseg;
        const size_t lb = align256((size_t)y.tiles * 256 * (y.wide ? 8 : 4));
        size_t o = 0;
        y.o_hist = o;
        o += align256((size_t)y.nseg * D * 256 * 8);
        y.o_done = o;
        o += align256((size_t)y.nseg * 4);
        y.o_ticket = o;
        o += 256;
        y.o_misc = o;  // most passes, counters, totals
        o += 256;
        y.o_hits = o;
        o += align256(sampled ? (size_t)y.nseg * RX_TRY * 4 : 0);
        y.o_tab = o;
        o += align256(sampled ? (size_t)many * RX_TRY * RX_SLOTS * 4 : 0);
        y.o_flags = o;
        o += align256((size_t)y.fixes);
        y.o_lb0 = o;
        o += lb;
        y.zero_bytes = o;  // everything up to here starts as zeros
        y.o_lb1 = o;
        o += lb;
        y.o_plan = o;
        o += align256((size_t)y.nseg * sizeof(RxPlan));
        y.o_at = o;
        o += align256((size_t)extra * sizeof(RxSegAt));
        y.o_tile = o;
        o += align256(extra ? (size_t)y.tiles * 4 : 0);
        y.o_chunk = o;
        o += align256(extra ? (size_t)y.chunks * 4 : 0);
        y.o_fix = o;
        o += align256(extra ? (size_t)y.fixes * 4 : 0);
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
        const unsigned grid = (unsigned)std::min<int64_t>(y.tiles, (int64_t)grid_sms * SH::CTAS);
        CT* l0 = (CT*)(ws + y.o_lb0);
        CT* l1 = (CT*)(ws + y.o_lb1);
        for (int i = 0; i < D; i++) {
            ProfScope ps_("radix_pass", s);
            launch_next(fp, grid, SH::NT, sb, s, A, i, (i & 1) ? l1 : l0, (i & 1) ? l0 : l1);
        }
        return cudaGetLastError();
    }

    template <int XF, typename CT>
    static cudaError_t passes(const SortArgs& a, const Layout& y, const RxArgs<K>& A, char* ws, int grid_sms)
    {
        cudaStream_t s = a.stream;
        cudaError_t e;
        if (y.nseg > 1) {
            ProfScope ps_("radix_segments", s);
            launch_next(k_rx_at<1024, K>, 1, 1024, 0, s, A);
            launch_next(k_rx_lists<K>, (unsigned)((y.nseg + 7) / 8), 256, 0, s, A);
        }
        if constexpr (std::is_same<K, Rec>::value) {
            ProfScope ps_("radix_descents", s);
            const int64_t g = (A.in.n0 + 4095) / 4096;
            launch_next(k_rx_descents<512>, (unsigned)std::min<int64_t>(g, grid_sms * 4), 512, 0, s, A.a.p, A.in.n0, A.descents);
        }
        if constexpr (D > 4) {
            ProfScope ps_("radix_sample", s);
            const unsigned z = (unsigned)std::min<int64_t>((y.S + 127) / 128, y.nseg == 1 ? 512 : 16);
            launch_next(k_rx_sample<K, XF>, dim3((unsigned)y.nseg, RX_TRY, z), 128, 0, s, A);
        }
        auto fc = k_rx_count<CNT, G, K, XF>;
        const size_t cb = (size_t)G * 4096 * 4;
        if ((e = smem_attr(fc, cb)) != cudaSuccess) return e;
        {
            ProfScope ps_("radix_count", s);
            launch_next(fc, dim3((unsigned)y.chunks, D / G), CNT, cb, s, A);
        }
        if (std::is_same<CT, uint32_t>::value && y.T == C::Small::T)
            e = digits<XF, uint32_t, typename C::Small>(y, A, ws, grid_sms, s);
        else if (std::is_same<CT, uint32_t>::value && y.T == C::Mid::T)
            e = digits<XF, uint32_t, typename C::Mid>(y, A, ws, grid_sms, s);
        else
            e = digits<XF, CT, typename C::Large>(y, A, ws, grid_sms, s);
        if (e != cudaSuccess) return e;
        if constexpr (D > 4) {
            {
                auto ff = k_rx_fix<K, XF>;
                constexpr size_t fb = sizeof(K) * (FT + 2 * FL + 1) + 2 * (FT / 2 + 2);
                if ((e = smem_attr(ff, fb)) != cudaSuccess) return e;
                ProfScope ps_("radix_fix", s);
                launch_next(ff, (unsigned)y.fixes, FN, fb, s, A);
            }
            auto fl = k_rx_long<K, XF, CT>;
            const size_t lb = std::max(TileBuf<K, 8>::type::bytes(FT), (size_t)(16 * 256 * 4 + 256 * 8 + 256 * 4 + 64));
            // the digit table (at most 1.5 rows of 1 KiB per LONG_T keys) and the list (two
            // entries per fix tile) share the look-back tables (two rows per tile)
            static_assert(2048.0 / C::Large::T >= 1.5 * 1024 / LONG_T + 2.0 * sizeof(RxBad) / FT &&
                              2048.0 / C::Mid::T >= 1.5 * 1024 / LONG_T + 2.0 * sizeof(RxBad) / FT &&
                              2048.0 / C::Small::T >= 1.5 * 1024 / LONG_T + 2.0 * sizeof(RxBad) / FT,
                          "the digit table and the list fit the look-back tables");
            if ((e = smem_attr(fl, lb)) != cudaSuccess) return e;
            ProfScope ps_("radix_long", s);
            launch_next(fl, (unsigned)grid_sms * LONG_CTAS, 512, lb, s, A);
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
        A.first = A.last = A.a;
        A.in.base = a.inst_base;
        A.in.n = a.inst_n;
        A.in.count = a.n_inst;
        A.in.n0 = a.n;
        A.nseg = y.nseg;
        A.iptr = std::is_same<K, Rec>::value ? nullptr : (K* const*)a.inst_ptrs;
        A.hist = (unsigned long long*)(ws + y.o_hist);
        A.plan = (RxPlan*)(ws + y.o_plan);
        A.done = (unsigned*)(ws + y.o_done);
        A.ticket = (unsigned*)(ws + y.o_ticket);
        A.T = y.T;
        A.chunk = y.chunk;
        A.sampled = D > 4;
        A.one = RxSegAt{0, 0, 0, (int)y.S, rx_lead(a.inst_base ? a.n_max : a.n), 0};
        A.ntiles1 = y.tiles;
        A.at = (RxSegAt*)(ws + y.o_at);
        A.tile_seg = (int*)(ws + y.o_tile);
        A.chunk_seg = (int*)(ws + y.o_chunk);
        A.fix_seg = (int*)(ws + y.o_fix);
        A.maxpass = (int*)(ws + y.o_misc);
        A.nflag = (unsigned*)(ws + y.o_misc + 4);
        A.total = (int64_t*)(ws + y.o_misc + 8);
        A.descents = (unsigned*)(ws + y.o_misc + 32);
        A.bads = (unsigned*)(ws + y.o_misc + 64);
        A.hits = (unsigned*)(ws + y.o_hits);
        A.tab = (unsigned*)(ws + y.o_tab);
        A.flags = (uint8_t*)(ws + y.o_flags);
        // the look-back tables serve k_rx_long once the passes are over
        const size_t list = align256((size_t)y.fixes * 2 * sizeof(RxBad));
        A.dtab = ws + y.o_lb0;
        A.rows = (unsigned)std::min<size_t>((y.o_plan - y.o_lb0 - list) / (y.wide ? 2048 : 1024), 0x7FFFFFFF);
        A.bad = (RxBad*)(ws + y.o_plan - list);
        A.spins = radix_spins();
        A.err = a.err ? a.err : (unsigned*)(ws + y.o_misc + 40);
        A.keep = a.keep_order_keys;
        return y.wide ? passes<XF, uint64_t>(a, y, A, ws, sms) : passes<XF, uint32_t>(a, y, A, ws, sms);
    }

    // ws == nullptr: the workspace comes from the pool; otherwise cap bytes at
    // ws are used and nothing is allocated (PS_ERR_INVALID_ARG if too few).
    static int run(const SortArgs& a, char* ws = nullptr, size_t cap = 0)
    {
        const Layout y = layout(a);
        char* own = nullptr;
        if (ws) {
            if (y.total > cap) return PS_ERR_INVALID_ARG;
        } else {
            const int rc = ws_alloc((void**)&own, y.total, a.stream);
            if (rc != PS_OK) return rc;
            ws = own;
        }
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
        if (own) ws_free(own, a.stream);
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

// launch_impl.cuh -- definitions of Launch<ST>; included by exactly one
// translation unit per storage type.
#pragma once

#include "kernels.cuh"
#include "launch.h"

namespace lbm {

template <typename ST, typename IXE, bool SNAP>
static cudaError_t launch_sc(const KP &p, int face, int odd, const Bufs &b, dim3 grd, dim3 blk, cudaStream_t st,
                             const SnapOut &snap) {
    // blocks resident at once: 7 of 128 threads an SM (72 registers)
    const int early = b.sms * (896 / (int)(blk.x * blk.y));
    const int *jm = p.skip_deep ? b.jmax : nullptr;
    ST *F = (ST *)b.F, *G = (ST *)b.G;
    if (face == 0) {
        if (odd) return launch_step_kernel(k_odd<ST, 0, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.nb_next, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm, early, b.s, snap);
        else return launch_step_kernel(k_even<ST, 0, IXE, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, jm, early, b.s, snap);
    } else {
        if (odd) return launch_step_kernel(k_odd<ST, 1, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.nb_next, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm, early, b.s, snap);
        else return launch_step_kernel(k_even<ST, 1, IXE, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, jm, early, b.s, snap);
    }
}

#ifndef LBM_PAIR_ODD_IX
#define LBM_PAIR_ODD_IX unsigned
#endif
template <typename ST, typename IX, int LIN, bool SNAP>
static cudaError_t launch_sc_pair_early(const KP &p, int face, int odd, const Bufs &b, dim3 grd, dim3 blk,
                                        cudaStream_t st, const SnapOut &snap) {
    const int early = b.sms * (pair_min_blocks<ST>() * 128 / (int)(blk.x * blk.y));  // blocks resident at once
    const int *jm = p.skip_deep ? b.jmax : nullptr;
    ST *F = (ST *)b.F, *G = (ST *)b.G;
    if (face == 0) {
        if (odd) return launch_step_kernel(k_odd_pair_early<ST, 0, IX, LIN, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.nb_next, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm, early, b.s, snap);
        else return launch_step_kernel(k_even_pair_early<ST, 0, IX, LIN, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, jm, early, b.s, snap);
    } else {
        if (odd) return launch_step_kernel(k_odd_pair_early<ST, 1, IX, LIN, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.nb_next, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm, early, b.s, snap);
        else return launch_step_kernel(k_even_pair_early<ST, 1, IX, LIN, SNAP>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, jm, early, b.s, snap);
    }
}

// An even nx: two nodes per thread (k_even_pair / k_odd_pair, or their early
// forms), the grid's x extent covering nx / 2 threads.
template <typename ST, typename IXE, typename IXO, int LIN>
static cudaError_t launch_sc_pair(const KP &p, int face, int odd, const Bufs &b, dim3 blk, cudaStream_t st,
                                  const SnapOut *snap) {
    const int *jm = p.skip_deep ? b.jmax : nullptr;
    ST *F = (ST *)b.F, *G = (ST *)b.G;
    KP half_x = p;
    half_x.nx = p.nx / 2;
    const dim3 grd = k1_grid(half_x, blk, face, b.k1_height, LIN);
    if constexpr (sizeof(ST) == 4 && sizeof(IXE) == 4) {
        if (b.early_pairs) {
            if (snap) return launch_sc_pair_early<ST, IXE, LIN, true>(p, face, odd, b, grd, blk, st, *snap);
            return launch_sc_pair_early<ST, IXE, LIN, false>(p, face, odd, b, grd, blk, st, SnapOut());
        }
    }
    if (face == 0) {
        if (odd) return launch_step_kernel(k_odd_pair<ST, 0, IXO, LIN>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm);
        else return launch_step_kernel(k_even_pair<ST, 0, IXE, LIN>, grd, blk, st, b.plain, p, F, G, b.js, b.nb, b.gpost, jm);
    } else {
        if (odd) return launch_step_kernel(k_odd_pair<ST, 1, IXO, LIN>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb, b.gpost, b.thw_rd, b.thw_wr, *b.lk, jm);
        else return launch_step_kernel(k_even_pair<ST, 1, IXE, LIN>, grd, blk, st, b.plain, p, F, G, b.js, b.nb, b.gpost, jm);
    }
}

// The even step indexes in 32 bits whenever every index of the 19 direction
// arrays of F fits (19 ld < 2^32: cavities up to about 2.2e8 nodes), else in
// 64 bits (FP16 storage 2% faster at 256^3; the odd step ran slower with
// 32-bit indices, 0.258 against 0.245 ms in FP32, and keeps 64-bit ones).
template <typename ST>
bool Launch<ST>::snapshots(const KP &p, const Bufs &b) {
    const bool pairs = b.pairs && p.nx % 2 == 0;
    return !p.cond && !(pairs && !(b.early_pairs && sizeof(ST) == 4)) && 19LL * p.ld < (1LL << 32);
}

template <typename ST>
cudaError_t Launch<ST>::stream_collide(const KP &p, int face, int odd, const Bufs &b, dim3 blk, cudaStream_t st,
                                       const SnapOut *snap) {
    if (p.cond) return LaunchCond<ST>::stream_collide(p, face, odd, b, blk, st);
    if (b.pairs && p.nx % 2 == 0) {
        if (19LL * p.ld < (1LL << 32)) {
            if (b.linear) return launch_sc_pair<ST, unsigned, LBM_PAIR_ODD_IX, 1>(p, face, odd, b, blk, st, snap);
            return launch_sc_pair<ST, unsigned, LBM_PAIR_ODD_IX, 0>(p, face, odd, b, blk, st, snap);
        }
        return launch_sc_pair<ST, long long, long long, 0>(p, face, odd, b, blk, st, nullptr);
    }
    const dim3 grd = k1_grid(p, blk, face, b.k1_height, b.linear);
    if (snap) return launch_sc<ST, unsigned, true>(p, face, odd, b, grd, blk, st, *snap);
    if (19LL * p.ld < (1LL << 32)) return launch_sc<ST, unsigned, false>(p, face, odd, b, grd, blk, st, SnapOut());
    return launch_sc<ST, long long, false>(p, face, odd, b, grd, blk, st, SnapOut());
}

template <typename ST>
cudaError_t Launch<ST>::front(const KP &p, int face, int inflight, int move, const Bufs &b, cudaStream_t st) {
    if (p.cond) return LaunchCond<ST>::front(p, face, inflight, move, b, st);
    const dim3 blk(b.cblk), grd = col_grid(p.ncols, b.cblk);
    ST *F = (ST *)b.F;
    const ST *G = (const ST *)b.G;
    if (face == 0)
        return launch_step_kernel(k_front<ST, 0>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb_next, b.s, b.s_next, b.gpost, b.thw_wr, inflight, move, b.status, b.jmax, b.jmax_host);
    return launch_step_kernel(k_front<ST, 1>, grd, blk, st, b.plain, p, F, G, b.js, b.js_next, b.nb_next, b.s, b.s_next, b.gpost, b.thw_wr, inflight, move, b.status, b.jmax, b.jmax_host);
}

template <typename ST>
cudaError_t Launch<ST>::macro(const KP &p, int face, int inflight, const Bufs &b, float *T, float *u, cudaStream_t st) {
    dim3 blk = node_block(p), grd = node_grid(p, blk);
    const ST *F = (const ST *)b.F, *G = (const ST *)b.G;
    if (face == 0) k_macro<ST, 0><<<grd, blk, 0, st>>>(p, F, G, b.js, b.js_next, b.thw_rd, inflight, T, u);
    else k_macro<ST, 1><<<grd, blk, 0, st>>>(p, F, G, b.js, b.js_next, b.thw_rd, inflight, T, u);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::state_out(const KP &p, int face, int inflight, const Bufs &b, float *f, float *g, cudaStream_t st) {
    dim3 blk = node_block(p), grd = node_grid(p, blk);
    const ST *F = (const ST *)b.F, *G = (const ST *)b.G;
    if (face == 0) k_state_out<ST, 0><<<grd, blk, 0, st>>>(p, F, G, b.js, b.js_next, b.nb, b.thw_rd, inflight, f, g);
    else k_state_out<ST, 1><<<grd, blk, 0, st>>>(p, F, G, b.js, b.js_next, b.nb, b.thw_rd, inflight, f, g);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::set_fronts(const KP &p, const Bufs &b, const double *s_in, double *s, int *js, cudaStream_t st) {
    k_set_fronts<<<col_grid(p.ncols, 128), 128, 0, st>>>(s_in, p.ncols, p.H, s, js, b.jmax, b.jmax_host);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::state_in(const KP &p, int face, const Bufs &b, const float *f, const float *g, cudaStream_t st) {
    dim3 blk = node_block(p), grd = node_grid(p, blk);
    ST *F = (ST *)b.F, *G = (ST *)b.G;
    if (face == 0) k_state_in<ST, 0><<<grd, blk, 0, st>>>(p, F, G, b.js, f, g);
    else k_state_in<ST, 1><<<grd, blk, 0, st>>>(p, F, G, b.js, f, g);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::init(const KP &p, int face, const Bufs &b, const float *Tprof, cudaStream_t st) {
    dim3 blk = node_block(p), grd = node_grid(p, blk);
    ST *F = (ST *)b.F, *G = (ST *)b.G;
    if (face == 0) k_init<ST, 0><<<grd, blk, 0, st>>>(p, F, G, b.js, Tprof);
    else k_init<ST, 1><<<grd, blk, 0, st>>>(p, F, G, b.js, Tprof);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::totals(const KP &p, int face, int inflight, const Bufs &b, double *part, int nparts,
                               double t, double *out, cudaStream_t st) {
    const ST *F = (const ST *)b.F, *G = (const ST *)b.G;
    const int col_tiles = (p.ncols + 255) / 256;
    const long long tiles = (long long)col_tiles * ((p.H + kTotalsRun - 1) / kTotalsRun);
    const int blocks = (int)(tiles < nparts ? tiles : nparts);
    if (face == 0)
        k_totals_part<ST, 0><<<blocks, 256, 0, st>>>(p, F, G, b.js, b.js_next, b.s, b.thw_rd, b.thw_nu, inflight,
                                                     b.nu_scale, part);
    else
        k_totals_part<ST, 1><<<blocks, 256, 0, st>>>(p, F, G, b.js, b.js_next, b.s, b.thw_rd, b.thw_nu, inflight,
                                                     b.nu_scale, part);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_totals_final<<<1, 256, 0, st>>>(part, blocks, p.ncols, (double)p.H, t, out);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t Launch<ST>::nusselt(const KP &p, int face, int inflight, const Bufs &b, cudaStream_t st) {
    const dim3 blk(b.cblk), grd = col_grid(p.ncols, b.cblk);
    const ST *G = (const ST *)b.G;
    if (face == 0) k_nusselt<ST, 0><<<grd, blk, 0, st>>>(p, G, b.thw_nu, inflight, b.nu_scale, b.nu);
    else k_nusselt<ST, 1><<<grd, blk, 0, st>>>(p, G, b.thw_nu, inflight, b.nu_scale, b.nu);
    return cudaGetLastError();
}

}  // namespace lbm

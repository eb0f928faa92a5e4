// launch.h -- host-side launchers of the kernels, one instantiation per
// storage type (k_f32.cu: float, k_f16.cu: __half).  Internal to the library.
#pragma once

#include <cuda_runtime.h>

#include "lbm_core.cuh"

namespace lbm {

struct Bufs {
    void *F, *G;                 // shifted distributions, 19 and 7 arrays of ld elements
    const int *js;               // liquid-node count per column (current flags)
    int *js_next;
    const int *nb;               // 3x3 min/max of js (min << 16 | max), current
    int *nb_next;
    const double *s;             // front per column (current)
    double *s_next;
    float *gpost;                // ghost-node post-collision g, 7 x ncols
    const float *thw_rd, *thw_wr;
    int *status;                 // page-locked: the front status, set on an error
    const Links *lk;             // interior link offsets of the odd step
    int cblk;                    // threads per block of the per-column kernels (col_block)
    int sms;                     // SMs of the device
    int *jmax;                   // running maximum of the liquid counts (k_front), or null
    int *jmax_host;              // its copy in page-locked host memory
    int k1_height;               // the stream-collide grid covers heights < k1_height (the rest is deep solid)
    const float *thw_nu;         // heated-wall field of the last streaming (Nusselt number)
    double *nu;                  // per-column Nusselt numbers (ncols)
    double nu_scale;             // H / (alpha (Th - Tm))
    float *spost;                // solid-side ghost populations, 7 x ncols (heat conduction in the solid)
    int pairs;                   // stream-collide with two nodes per thread (even nx)
    int linear;                  // stream-collide blocks of consecutive columns (k1_linear)
    int early_pairs;             // ... with the first wave's loads before the wait (FP32 storage, middle sizes)
    int plain;                   // launch without programmatic serialization (launch_step_kernel)
};

// Where a step leaves the natural-layout snapshot of the state it starts from
// (FP32: fh of 19 directions, zero at solid nodes, then gh of 7, each of N
// nodes in rows of nx and planes of ny rows: the heights below `heights`
// only), and the columns' fronts, liquid counts and 3x3 bounds.
struct SnapOut {
    float *out;
    double *s;
    int *js, *nb;
    long long N;
    int ny, heights;
};

// The stream-collide and front kernels with heat conduction in the solid
// (KP::cond), in a translation unit of their own (k_cond.cu); Launch
// forwards to them.
template <typename ST> struct LaunchCond {
    static cudaError_t stream_collide(const KP &p, int face, int odd, const Bufs &b, dim3 blk, cudaStream_t st);
    static cudaError_t front(const KP &p, int face, int inflight, int move, const Bufs &b, cudaStream_t st);
};

template <typename ST> struct Launch {
    // snap (may be null): also write the snapshot of the state the step starts
    // from; only where snapshots(p, b).
    static cudaError_t stream_collide(const KP &p, int face, int odd, const Bufs &b, dim3 blk, cudaStream_t st,
                                      const SnapOut *snap = nullptr);
    static bool snapshots(const KP &p, const Bufs &b);
    static cudaError_t front(const KP &p, int face, int inflight, int move, const Bufs &b, cudaStream_t st);
    static cudaError_t macro(const KP &p, int face, int inflight, const Bufs &b, float *T, float *u, cudaStream_t st);
    static cudaError_t state_out(const KP &p, int face, int inflight, const Bufs &b, float *f, float *g, cudaStream_t st);
    static cudaError_t set_fronts(const KP &p, const Bufs &b, const double *s_in, double *s, int *js, cudaStream_t st);
    static cudaError_t state_in(const KP &p, int face, const Bufs &b, const float *f, const float *g, cudaStream_t st);
    static cudaError_t init(const KP &p, int face, const Bufs &b, const float *Tprof, cudaStream_t st);
    static cudaError_t totals(const KP &p, int face, int inflight, const Bufs &b, double *part, int nparts,
                              double t, double *out, cudaStream_t st);
    static cudaError_t nusselt(const KP &p, int face, int inflight, const Bufs &b, cudaStream_t st);
};

// Threads per block of the per-column kernels (front and its adjoints): the largest of 128, 64 and 32 that still gives two blocks per
// SM, so that a small front (96 x 96 columns) spreads its FP64 arithmetic
// over all SMs instead of half of them.
inline int col_block(long long ncols, int sms) {
    for (int b = 128; b > 32; b >>= 1)
        if ((ncols + b - 1) / b >= 2LL * sms) return b;
    return 32;
}
inline dim3 col_grid(long long ncols, int b) { return dim3((unsigned)((ncols + b - 1) / b)); }

// Block shape for the per-node kernels: 128 threads, x-major.
// Width along x of a block of `block` threads: the power of two from 32 to
// min(block, 128) that leaves the fewest idle lanes over a row of nx nodes
// (the widest on a tie): 160 -> 32, 96 -> 32, 48 -> 64, 256 -> 128.
inline int block_width(int nx, int block) {
    int best = 32;
    long long best_waste = -1;
    for (int bx = 32; bx <= block && bx <= 128; bx *= 2) {
        const long long waste = (long long)((nx + bx - 1) / bx) * bx - nx;
        if (best_waste < 0 || waste <= best_waste) {
            best = bx;
            best_waste = waste;
        }
    }
    return best;
}
// Whether rows of nxt threads (nx, or nx / 2 with two nodes per thread) leave
// lanes idle in the fitted width: then the stream-collide's blocks take
// consecutive columns instead.  Us per step, rows against columns, front at
// 0.5 H: 71^3 13.7 / 12.6, 101x75x83 18.3 / 16.9, 100^3 24.4 / 22.0, 160^3 (80
// pairs a row) 81.1 / 78.3, 200^3 166.8 / 159.2, 200^3 with a conducting solid
// 196 / 186, FP16 100^3 22.0 / 19.4.  Rows that fit keep their blocks (FP16
// 160^3 55.0 / 56.9, 256^3 162 / 171; FP32 the same either way).
inline bool k1_linear(int nxt, int widest) {
    const int bx = block_width(nxt, widest);
    return nxt % bx != 0;
}
inline dim3 node_block(const KP &p) {
    const int bx = block_width(p.nx, 128);
    return dim3(bx, 128 / bx, 1);
}
inline dim3 node_grid(const KP &p, dim3 b) {
    return dim3((p.nx + b.x - 1) / b.x, (p.ny + b.y - 1) / b.y, p.nz);
}
// Grid of the stream-collide (k1_node): x tiles, the in-plane tiles, then
// the heights along the heating axis (slowest).
// Linear: blocks of 128 consecutive columns (b.x; pairs of them with p.nx
// halved), whatever rows they lie in.
inline dim3 k1_grid(const KP &p, dim3 b, int face, int height, int linear) {
    if (linear) {
        if (height < 1) height = 1;
        return dim3((unsigned)(((long long)p.nx * p.P2 + b.x - 1) / b.x), 1, height < p.H ? height : p.H);
    }
    const unsigned gx = (p.nx + b.x - 1) / b.x;
    if (height < 1) height = 1;
    if (face == 0) {
        const unsigned gz = (unsigned)((height + (int)b.y - 1) / (int)b.y), full = (p.ny + b.y - 1) / b.y;
        return dim3(gx, p.nz, gz < full ? gz : full);
    }
    return dim3(gx, (p.ny + b.y - 1) / b.y, (unsigned)(height < p.nz ? height : p.nz));
}

// node_grid cut to the heights a < abound along the heating axis (y for
// face 0, z for face 1).
inline dim3 node_grid_axial(const KP &p, dim3 b, int face, int abound) {
    dim3 g = node_grid(p, b);
    if (abound < 1) abound = 1;
    if (face == 0) {
        const unsigned gy = (unsigned)((abound + (int)b.y - 1) / (int)b.y);
        if (gy < g.y) g.y = gy;
    } else if ((unsigned)abound < g.z) {
        g.z = (unsigned)abound;
    }
    return g;
}

}  // namespace lbm

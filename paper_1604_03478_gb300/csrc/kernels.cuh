// kernels.cuh -- the device kernels of one time step and of the state I/O,
// templated on the storage type (float or __half) and the heated face.
//
// One step of the method (Li, Yang & Zhang, arXiv:1604.03478, section 2):
//   k_even / k_odd : fused stream + collide of f (D3Q19 MRT, Eqs. 1-3) and
//                    g (D3Q7 MRT, Eqs. 4-5), in place by the AA pattern, one
//                    node per thread (k_even_pair / k_odd_pair: two
//                    x-adjacent nodes per thread in packed FP32x2 arithmetic);
//   k_front        : interfacial tracking, Eq. 6, one thread per column (FP64
//                    fronts, FP32 gradient and speed), and the phase flip of
//                    the nodes the front crossed.
//
// AA pattern.  A step that starts from the natural layout (slot i of node x
// holds f_i(x), "even") reads and writes only node x: the post-collision
// f*_i goes to slot opp(i) of x.  The next step ("odd") pulls f_i(x) from
// slot opp(i) of x - e_i and pushes f*_i to slot i of x + e_i, which brings
// the layout back to natural.  Walls and liquid/solid links are handled on
// the odd step's reads and writes: a missing upstream node means halfway
// bounce-back (read slot i of x itself), a missing downstream node means the
// value stays at x in slot opp(i).  Every node reads and writes the same set
// of slots in a step, so the update is race-free in place.
//
// Between an even and an odd step the post-collision values are "in flight"
// (their streaming is deferred to the odd step).  If the front flips a node
// there, the odd step would read the in-flight values with the new flags;
// flip_column moves the value of every link between a flipped node and a node
// that was liquid to the slot where the new flags look for it, and a reader
// takes f = f^eq(1, 0) for a node that is liquid now and was not under the
// flags of the step before (the other of the two liquid-count buffers).
#pragma once

#include "launch.h"
#include "lbm_core.cuh"

namespace lbm {

// Programmatic dependent launch: the kernels of a step are launched so that
// the next one may be scheduled while the previous one drains; each waits
// for its predecessor's completion (and memory) before its first access,
// then lets its own successor be scheduled.  Both are no-ops for a kernel
// launched without the attribute.
__device__ __forceinline__ void step_launch_wait() {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
// How the kernels that call step_launch_wait are launched (the step's, the
// adjoint's): with programmatic stream serialization, but plainly (`plain`)
// after a kernel that is not one of them and writes what this one loads before
// its wait (a wall field, fronts, a restored state): such a kernel lets its
// successor start when its blocks have returned, which does not order its
// stores before loads that no wait precedes.
template <typename... KArgs, typename... Args>
static cudaError_t launch_step_kernel(void (*kern)(KArgs...), dim3 grd, dim3 blk, cudaStream_t st, int plain, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grd;
    cfg.blockDim = blk;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = plain ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// What a kernel may load before step_launch_wait: whatever its immediate
// predecessor does not write.  The predecessor let this kernel start only
// after its own wait, so everything before the predecessor is complete (after
// other kernels, which have no such wait, the launch is plain: see
// launch_step_kernel).  Such loads go to L2 (ld.global.cg): L1 may hold a line from before.  They and
// the wait are volatile, so the compiler keeps their order.
// After the wait, what the front update writes (js, nb, gpost, spost) is read
// by ordinary loads: never by __ldg and never through a const __restrict__
// parameter, which allow the non-coherent path and promise that nobody writes
// it while the grid lives, and its early blocks live while the front update
// still writes.  The same holds for the ensemble's kernel, which writes them
// itself.
__device__ __forceinline__ int ld_l2(const int *q) {
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];\n" : "=r"(v) : "l"(q));
    return v;
}
__device__ __forceinline__ int2 ld_l2(const int2 *q) {
    int2 v;
    asm volatile("ld.global.cg.v2.s32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(q));
    return v;
}
__device__ __forceinline__ float2 ld_l2(const float2 *q) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(q));
    return v;
}
__device__ __forceinline__ double ld_l2(const double *q) {
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];\n" : "=d"(v) : "l"(q));
    return v;
}
__device__ __forceinline__ float ld_l2(const float *q) {
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];\n" : "=f"(v) : "l"(q));
    return v;
}
__device__ __forceinline__ float ld_l2(const __half *q) {
    unsigned short v;
    asm volatile("ld.global.cg.u16 %0, [%1];\n" : "=h"(v) : "l"(q));
    return __half2float(__ushort_as_half(v));
}

template <int FACE> __device__ __forceinline__ long long off19(const KP &p, int i) {
    return (long long)ex(i) + (long long)ey(i) * p.nx + (long long)ez(i) * p.nx * p.ny;
}
template <int FACE> __device__ __forceinline__ long long off7(const KP &p, int i) {
    return (long long)tx(i) + (long long)ty(i) * p.nx + (long long)tz(i) * p.nx * p.ny;
}

// Element offsets of the odd step's interior links: from the table lk (a
// kernel parameter) when TAB, else from the extents.
template <int FACE, bool TAB> __device__ __forceinline__ long long fin_off(const KP &p, const Links *lk, int i) {
    return TAB ? lk->fin[i] : opp(i) * p.ld - off19<FACE>(p, i);
}
template <int FACE, bool TAB> __device__ __forceinline__ long long fout_off(const KP &p, const Links *lk, int i) {
    return TAB ? lk->fout[i] : i * p.ld + off19<FACE>(p, i);
}
template <int FACE, bool TAB> __device__ __forceinline__ long long gin_off(const KP &p, const Links *lk, int i) {
    return TAB ? lk->gin[i] : opp7(i) * p.ld - off7<FACE>(p, i);
}
template <int FACE, bool TAB> __device__ __forceinline__ long long gout_off(const KP &p, const Links *lk, int i) {
    return TAB ? lk->gout[i] : i * p.ld + off7<FACE>(p, i);
}

// Element base[c + off] with the index arithmetic done in IX: unsigned (32
// bits, for states whose every element index fits) or long long.  With
// 32-bit indices a link offset enters the address as one 32-bit add of a
// kernel-parameter operand.
template <typename IX, typename ST>
__device__ __forceinline__ ST *elem(ST *base, IX c, long long off) {
    return base + (IX)(c + (IX)off);
}

// Post-collision shifted g of a solid node: the ghost node (first solid node
// of its column) takes the populations prepared by k_front; deeper nodes are
// at rest at Tm (gh = w (Tm - Ts), zero with FP32 storage).
__device__ __forceinline__ void solid_post(const KP &p, bool ghost, const float *gpost, int col, float (&g)[7]) {
#pragma unroll
    for (int i = 0; i < 7; ++i) g[i] = ghost ? gpost[(long long)i * p.ncols + col] : w7(i) * p.dTms;
}

// A solid node at least two nodes above its column's first solid node and
// above every 3x3-neighbour column's first solid node ("deep") has only
// solid neighbours that are not ghost nodes.  Nothing reads its slots while
// it is deep, and one step before the front can reach it, it is no longer
// deep (the 3x3 maximum includes its own column), so with Tc = Tm (the cold
// wall then returns zero too) its update can be skipped exactly.
__device__ __forceinline__ bool deep_solid(const KP &p, int a, int nbv) {
    return p.skip_deep && a >= (nbv & 0xffff) + 2;
}

// ------------------------------------------------- conduction in the solid
// Bit i (1..6): the D3Q7 link leaving node x along t_i ends inside the
// cavity on a node of the other phase (liq: x is liquid).
template <int FACE>
__device__ __forceinline__ unsigned other_phase7(const KP &p, const int *js, int x, int y, int z,
                                                 bool liq) {
    unsigned m = 0;
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const int xn = x + tx(i), yn = y + ty(i), zn = z + tz(i);
        if (inside(p, xn, yn, zn) && (axial<FACE>(xn, yn, zn) < js[column<FACE>(p, xn, yn, zn)]) != liq)
            m |= 1u << i;
    }
    return m;
}

// With heat conduction in the solid, a population leaving node x towards a
// node of the other phase (bits of `other`) is not x's own post-collision
// value: it is the ghost population of x's column for the receiving phase
// when x is that ghost (ghost: the first solid node towards the liquid, with
// the liquid side's ghost populations gbuf; the last liquid node towards the
// solid, with the solid side's), else the rest state at Tm.
__device__ __forceinline__ void cross_phase(const KP &p, unsigned other, bool ghost, const float *gbuf,
                                            int col, float (&g)[7]) {
#pragma unroll
    for (int i = 1; i < 7; ++i)
        if ((other >> i) & 1u) g[i] = ghost ? gbuf[(long long)i * p.ncols + col] : w7(i) * p.dTms;
}

// ------------------------------------------------------------- even step
// COND: heat conduction in the solid (the solid collides its own g at u = 0
// and the links across the phase boundary carry the ghost or rest values of
// cross_phase; spost holds the solid side's ghost populations).
template <typename ST, int FACE, typename IX = long long, bool COND = false>
__device__ __forceinline__ void even_node(const KP &p, ST *__restrict__ F, ST *__restrict__ G, const int *js,
                                          const int *nb, const float *gpost, int x, int y,
                                          int z, const float *spost = nullptr) {
    const IX c = (IX)node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z);
    const int col = column<FACE>(p, x, y, z);
    const int jsc = js[col];
    float g[7];
    if (a < jsc) {
        float f[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) f[i] = Store<ST>::ld(elem<IX>(F, c, i * p.ld));
#pragma unroll
        for (int i = 0; i < 7; ++i) g[i] = Store<ST>::ld(elem<IX>(G, c, i * p.ld));
        collide(p, f, g);
#pragma unroll
        for (int i = 0; i < 19; ++i) Store<ST>::st_stream(elem<IX>(F, c, opp(i) * p.ld), f[i]);
        if (COND && a + 1 >= (nb[col] >> 16)) {
            const unsigned other = other_phase7<FACE>(p, js, x, y, z, true);
            if (other) cross_phase(p, other, a == jsc - 1, spost, col, g);
        }
    } else if (COND) {
#pragma unroll
        for (int i = 0; i < 7; ++i) g[i] = Store<ST>::ld(elem<IX>(G, c, i * p.ld));
        collide_solid(p, g);
        if (a <= (nb[col] & 0xffff)) {
            const unsigned other = other_phase7<FACE>(p, js, x, y, z, false);
            if (other) cross_phase(p, other, a == jsc, gpost, col, g);
        }
    } else {
        if (deep_solid(p, a, nb[col])) return;
        solid_post(p, a == jsc, gpost, col, g);
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) Store<ST>::st_stream(elem<IX>(G, c, opp7(i) * p.ld), g[i]);
}

// ---------------------------------------------------------- snapshots
__device__ __forceinline__ void snap_node(const KP &p, const SnapOut &o, int x, int y, int z, const float (&f)[19],
                                          const float (&g)[7]) {
    float *const at = o.out + (((long long)z * o.ny + y) * p.nx + x);
#pragma unroll
    for (int i = 0; i < 19; ++i) at[i * o.N] = f[i];
#pragma unroll
    for (int i = 0; i < 7; ++i) at[(19 + i) * o.N] = g[i];
}
__device__ __forceinline__ void snap_column(const SnapOut &o, int col, double s, int js, int nb) {
    o.s[col] = s;
    o.js[col] = js;
    o.nb[col] = nb;
}

// A pair's (N and the pair's index are even: 8-byte aligned).
__device__ __forceinline__ void snap_pair(const KP &p, const SnapOut &o, int x, int y, int z, const float2 (&f)[19],
                                          const float2 (&g)[7]) {
    float *const at = o.out + (((long long)z * o.ny + y) * p.nx + x);
#pragma unroll
    for (int i = 0; i < 19; ++i) *(float2 *)(at + i * o.N) = f[i];
#pragma unroll
    for (int i = 0; i < 7; ++i) *(float2 *)(at + (19 + i) * o.N) = g[i];
}
__device__ __forceinline__ void snap_pair_columns(const SnapOut &o, int col, const double *s, const int *js,
                                                  const int *nb) {
    snap_column(o, col, s[col], js[col], nb[col]);
    snap_column(o, col + 1, s[col + 1], js[col + 1], nb[col + 1]);
}
// The snapshot of a column's first solid node: fh = 0 and its g.
template <typename ST, int FACE>
__device__ __forceinline__ void snap_ghost(const KP &p, const ST *G, const float *thw, int x, int y, int z,
                                           bool inflight, const SnapOut &o);
// The snapshot of a node that is liquid or its column's first solid one.
template <typename ST, int FACE>
__device__ __forceinline__ void snap_any(const KP &p, const ST *F, const ST *G, const int *js, const int *js_old,
                                         const float *thw, int x, int y, int z, bool inflight, const SnapOut &o);

// Stream-collide grid: blocks of blockDim.x x blockDim.y nodes of one plane
// across the heating axis, with the height along that axis slowest
// (blockIdx.z), so that the blocks near the heated wall are dispatched
// first.  jmax (null: no bound) is the running maximum of the liquid counts,
// written by the previous front update: nodes two or more above every
// neighbouring count are deep solid and do nothing, so a block whose heights
// are all >= jmax + 3 returns at once.
// A grid of one block row (gridDim.y == blockDim.y == 1) is linear instead:
// consecutive threads take consecutive columns of one height, across the ends
// of rows, so that no lane idles whatever nx is (k1_linear in launch.h says
// when).
__device__ __forceinline__ bool k1_is_linear() { return gridDim.y == 1 && blockDim.y == 1; }
// Lowest height of a block of the stream-collide grid.
template <int FACE> __device__ __forceinline__ int k1_low() {
    return (int)blockIdx.z * (FACE == 0 ? (int)blockDim.y : 1);
}
// Whether the block is past the first `early_blocks` of the grid, the ones
// that are resident at once.
__device__ __forceinline__ bool k1_late(int early_blocks) {
    return (long long)(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x >= early_blocks;
}
template <int FACE>
__device__ __forceinline__ bool k1_node(const KP &p, int &x, int &y, int &z) {
    const int a0 = k1_low<FACE>();
    x = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (k1_is_linear()) {
        const int q = (int)((unsigned)x / (unsigned)p.nx);
        x -= q * p.nx;
        y = FACE == 0 ? a0 : q;
        z = FACE == 0 ? q : a0;
        return q < p.P2 && a0 < p.H;
    }
    if (FACE == 0) {
        y = a0 + (int)threadIdx.y;
        z = (int)blockIdx.y;
    } else {
        y = (int)(blockIdx.y * blockDim.y + threadIdx.y);
        z = (int)blockIdx.z;
    }
    return x < p.nx && y < p.ny;
}

// Resident blocks of 128 the stream-collide asks for: 8 (64 registers, a
// few bytes of spills) for FP16 storage, whose warps move half the bytes and
// need more of them in flight (+1.3%); none for FP32 (72 registers, 7
// blocks, no spills; forced to 8 it loses 1%).
template <typename ST> constexpr int k1_min_blocks() { return sizeof(ST) == 2 ? 8 : 0; }

// One node per thread.  These are the kernels of the smaller cavities, whose
// step is a chain of latencies, so the blocks that find a place while the
// front update of the step before still runs load a liquid node's
// populations before step_launch_wait: the front update writes slots of nodes
// that were solid only (flip_column), and a node that has just become liquid
// takes what it wrote after the wait.  The blocks that start later
// (early_blocks and on) find the wait over; they wait first and read the
// flags through L1, which their neighbours on the SM have filled: with their
// flags from L2 too, 128^3 with a thin layer ran 17.0 us a step, 96^3 18.8.
// A step, without and with the early loads: 32^3 8.0 -> 6.5 us, 128^3 thin
// layer 16.8 -> 16.5, 96^3 mid melt 18.6 -> 18.2, 101x75x83 19.6 -> 18.9.
//
// SNAP: the snapshot of the state the step starts from (the recomputation of
// the adjoint): the liquid nodes' populations, which the step has in
// registers, and the first solid node's g.
template <typename ST, int FACE, typename IX, bool SNAP>
__global__ void __launch_bounds__(128, SNAP ? 0 : k1_min_blocks<ST>()) k_even(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                              const int *js, const int *js_old, const int *nb,
                                              const float *gpost, const int *jmax, int early_blocks,
                                              const double *s, const __grid_constant__ SnapOut snap) {
    int x = 0, y = 0, z = 0, a = 0, col = 0, jso = 0;
    IX c = 0;
    float f[19], g[7];
    bool on = k1_node<FACE>(p, x, y, z);
    const bool late = k1_late(early_blocks);
    if (late) step_launch_wait();
    if (on) {
        c = (IX)node_index(p, x, y, z);
        a = axial<FACE>(x, y, z);
        col = column<FACE>(p, x, y, z);
        const int jm = jmax ? (late ? *jmax : ld_l2(jmax)) : 1 << 29;
        jso = late ? js_old[col] : ld_l2(js_old + col);
        on = k1_low<FACE>() < jm + 3;
        if (a < jso) {
#pragma unroll
            for (int i = 0; i < 19; ++i) f[i] = ld_l2(elem<IX>(F, c, i * p.ld));
#pragma unroll
            for (int i = 0; i < 7; ++i) g[i] = ld_l2(elem<IX>(G, c, i * p.ld));
        }
    }
    if (!late) step_launch_wait();
    if (!on) return;
    const int jsc = js[col];
    if (SNAP && a == 0) snap_column(snap, col, s[col], jsc, nb[col]);
    if (a < jsc) {
        if (a >= jso) {
#pragma unroll
            for (int i = 0; i < 19; ++i) f[i] = ld_l2(elem<IX>(F, c, i * p.ld));
#pragma unroll
            for (int i = 0; i < 7; ++i) g[i] = ld_l2(elem<IX>(G, c, i * p.ld));
        }
        if (SNAP) snap_node(p, snap, x, y, z, f, g);
        collide(p, f, g);
#pragma unroll
        for (int i = 0; i < 19; ++i) Store<ST>::st_stream(elem<IX>(F, c, opp(i) * p.ld), f[i]);
    } else {
        if (deep_solid(p, a, nb[col])) return;
        if (SNAP && a == jsc) snap_ghost<ST, FACE>(p, G, nullptr, x, y, z, false, snap);
        solid_post(p, a == jsc, gpost, col, g);
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) Store<ST>::st_stream(elem<IX>(G, c, opp7(i) * p.ld), g[i]);
}

// The even step with heat conduction in the solid (every node updated).
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_even_cond(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                                   const int *js, const int *nb,
                                                   const float *gpost, const float *spost) {
    step_launch_wait();
    int x, y, z;
    if (k1_node<FACE>(p, x, y, z)) even_node<ST, FACE, long long, true>(p, F, G, js, nb, gpost, x, y, z, spost);
}


// -------------------------------------------------------------- odd step
// Liquid counts of the 3x3 columns around column (pp, q), 0 outside the
// cavity; entry (dq + 1) * 3 + dp + 1.  FIXED: in a kernel during which nobody
// writes them (read-outs, the adjoint's node kernel), through the read-only
// path (fields and totals of a 256^3 state 376 us, else 390).  The front update
// of a lone cavity is one too, not the ensemble's (SPEC, see front_column).
template <bool FIXED = false>
__device__ __forceinline__ void load_js9(const KP &p, const int *js, int pp, int q, int (&js9)[9]) {
#pragma unroll
    for (int dq = -1; dq <= 1; ++dq)
#pragma unroll
        for (int dp = -1; dp <= 1; ++dp) {
            const int p2 = pp + dp, q2 = q + dq;
            const bool in = (unsigned)p2 < (unsigned)p.P1 && (unsigned)q2 < (unsigned)p.P2;
            js9[(dq + 1) * 3 + dp + 1] = in ? (FIXED ? __ldg(js + q2 * p.P1 + p2) : js[q2 * p.P1 + p2]) : 0;
        }
}

// load_js9 by loads that may stand before step_launch_wait.
__device__ __forceinline__ void load_js9_l2(const KP &p, const int *js, int pp, int q, int (&js9)[9]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int p2 = pp + k % 3 - 1, q2 = q + k / 3 - 1;
        const bool in = (unsigned)p2 < (unsigned)p.P1 && (unsigned)q2 < (unsigned)p.P2;
        js9[k] = in ? ld_l2(js + q2 * p.P1 + p2) : 0;
    }
}

// Bit i (1..18) of the link mask: node x - e_i is inside and liquid, i.e.
// f_i streams in from there (else halfway bounce-back).  Since x + e_i =
// x - e_opp(i), bit opp(i) tells whether f*_i streams out to x + e_i.
// From the counts js9 of the node's 3x3 columns and its height a.
template <int FACE>
__device__ __forceinline__ unsigned link_mask9(const int (&js9)[9], int a) {
    unsigned m = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        // the upstream node x - e_i: in-plane column offset and height
        const int dp = -ex(i), dq = FACE == 0 ? -ez(i) : -ey(i), da = FACE == 0 ? -ey(i) : -ez(i);
        const int an = a + da;
        if (an >= 0 && an < js9[(dq + 1) * 3 + dp + 1]) m |= 1u << i;
    }
    return m;
}

// Liquid counts of the twelve columns around those of a pair (the 3x3 columns
// of both, pp - 1 .. pp + 2 by q - 1 .. q + 1), 0 outside the cavity; entry
// (dq + 1) * 4 + dp + 1.
__device__ __forceinline__ void load_js12(const KP &p, const int *js, int pp, int q, int (&c)[12]) {
#pragma unroll
    for (int dq = -1; dq <= 1; ++dq)
#pragma unroll
        for (int dp = -1; dp <= 2; ++dp) {
            const int p2 = pp + dp, q2 = q + dq;
            const bool in = (unsigned)p2 < (unsigned)p.P1 && (unsigned)q2 < (unsigned)p.P2;
            c[(dq + 1) * 4 + dp + 1] = in ? js[q2 * p.P1 + p2] : 0;
        }
}
// Smallest (over columns inside the cavity) and largest of them.
__device__ __forceinline__ void range_js12(const KP &p, const int (&c)[12], int pp, int q, int &mn, int &mx) {
    mn = 1 << 15;
    mx = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int dp = k % 4 - 1, dq = k / 4 - 1;
        const bool in = (unsigned)(pp + dp) < (unsigned)p.P1 && (unsigned)(q + dq) < (unsigned)p.P2;
        mn = in && c[k] < mn ? c[k] : mn;
        mx = c[k] > mx ? c[k] : mx;
    }
}
// The 3x3 counts (load_js9) of the pair's node `lane` (0 or 1).
__device__ __forceinline__ void js9_of_js12(const int (&c)[12], int lane, int (&js9)[9]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) js9[k] = lane ? c[k / 3 * 4 + k % 3 + 1] : c[k / 3 * 4 + k % 3];
}

// Bit i (1..6): node x - t_i is inside (else the link crosses a wall).
__device__ __forceinline__ unsigned inside_mask(const KP &p, int x, int y, int z) {
    unsigned m = 0;
#pragma unroll
    for (int i = 1; i < 7; ++i)
        if (inside(p, x - tx(i), y - ty(i), z - tz(i))) m |= 1u << i;
    return m;
}

// Wall rule for a D3Q7 population leaving along link direction `dir`
// across a wall: adiabatic bounce-back keeps it, the isothermal walls return
// -v + 2 w (Tw - Ts) (anti-bounce-back, shifted populations).
template <int FACE>
__device__ __forceinline__ float wall_value(const KP &p, int dir, float v, float Th_col) {
    const int w = wall_of_link<FACE>(dir);
    return w == 3 ? v : -v + 2.0f * w7(dir) * ((w == 1 ? Th_col : p.Tc) - p.Ts);
}

// Across an x wall (x = 0 for e_x = +1 upstream, x = nx - 1 for e_x = -1):
// the only walls a warp's nodes (32 consecutive x at one height and plane)
// do not all share.
__device__ __forceinline__ bool xwall(int ex_up, bool xlo, bool xhi) {
    return ex_up > 0 ? xlo : (ex_up < 0 ? xhi : false);
}

// TAB: take the interior link offsets from the precomputed tables of KP
// (kernel parameters: constant-bank operands); false computes them from the
// extents, which keeps them out of registers when KP lives in shared memory.
//
// Fast path: a liquid node off the walls of the heating axis and of the
// other in-plane axis and at least one node below the lowest first-solid
// node of its 3x3 neighbour columns (by the bounds of nb, which may be two
// low, else by the counts themselves, which the general path needs for its
// link mask anyway), so that every link streams except those
// across an x wall, which bounce back (no-slip for f, adiabatic for g).  The
// x walls are taken by selects inside the fast path, so that the warps that
// hold x = 0 or x = nx - 1 do not split between two paths.
//
// COND: heat conduction in the solid (see even_node).
//
// known: the node's 3x3 liquid counts where the caller has them, else null.
//
// js_old: the liquid counts the in-flight values were produced under.  A node
// that has become liquid since (never on the fast path: the count bounds nb
// are at most the old counts less one) starts from fh = 0.
template <typename ST, int FACE, bool TAB = true, bool COND = false>
__device__ __forceinline__ void odd_node(const KP &p, const Links *lk, ST *__restrict__ F, ST *__restrict__ G, const int *js,
                                         const int *js_old, const int *nb, const float *gpost,
                                         const float *__restrict__ thw_rd, const float *__restrict__ thw_wr, int x,
                                         int y, int z, const float *spost = nullptr,
                                         const int *known = nullptr) {
    const long long c = node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z);
    const int col = column<FACE>(p, x, y, z);
    const int jsc = js[col];
    const int nbv = nb[col];
    const int q = FACE == 0 ? z : y, nq = FACE == 0 ? p.nz : p.ny;
    const bool off_qa = q >= 1 && q <= nq - 2 && a >= 1 && a <= p.H - 2;
    const bool off_walls = off_qa && x >= 1 && x <= p.nx - 2;
    const bool xlo = x == 0, xhi = x == p.nx - 1;
    ST *const Fc = F + c;
    ST *const Gc = G + c;
    float g[7];
    if (a < jsc) {
        bool fast = off_qa && a + 1 < (nbv >> 16);
        float f[19];
        unsigned lm = 0x7fffeu, im = 0x7eu;
        if (!fast) {
            int js9[9];
            if (known) {
#pragma unroll
                for (int k = 0; k < 9; ++k) js9[k] = known[k];
            } else {
                load_js9(p, js, x, q, js9);
            }
            lm = link_mask9<FACE>(js9, a);
            im = inside_mask(p, x, y, z);
            // off the walls a full mask, but for the links across an x wall
            // (which read count 0), is the interior
            if (off_qa) {
                unsigned need = 0x7fffeu;
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (xwall(ex(i), xlo, xhi)) need &= ~(1u << i);
                fast = (lm & need) == need;
            }
        }
        if (fast) {
#pragma unroll
            for (int i = 0; i < 19; ++i) f[i] = Store<ST>::ld(Fc + fin_off<FACE, TAB>(p, lk, i));
#pragma unroll
            for (int i = 0; i < 7; ++i) g[i] = Store<ST>::ld(Gc + gin_off<FACE, TAB>(p, lk, i));
            // Across an x wall the pull above read the neighbouring row's
            // node instead (an in-bounds element of the same direction array:
            // the node is off the walls of the other two axes); bounce-back
            // replaces it with the value parked in the node's own slot i
            // (no-slip for f, adiabatic for g).
            if (xlo | xhi) {
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (xwall(ex(i), xlo, xhi)) f[i] = Store<ST>::ld(Fc + i * p.ld);
#pragma unroll
                for (int i = 1; i < 7; ++i)
                    if (xwall(tx(i), xlo, xhi)) g[i] = Store<ST>::ld(Gc + i * p.ld);
            }
        } else {
            const float th_rd = __ldg(thw_rd + col);
            const bool was_liquid = a < js_old[col];
            f[0] = Store<ST>::ld(Fc);
#pragma unroll
            for (int i = 1; i < 19; ++i)  // else bounce-back: f*_opp(i) parked in slot i
                f[i] = Store<ST>::ld(((lm >> i) & 1u) ? Fc + fin_off<FACE, TAB>(p, lk, i) : Fc + i * p.ld);
            if (!was_liquid) {
#pragma unroll
                for (int i = 0; i < 19; ++i) f[i] = 0.0f;
            }
            g[0] = Store<ST>::ld(Gc);
#pragma unroll
            for (int i = 1; i < 7; ++i) {
                const bool in = (im >> i) & 1u;
                const float v = Store<ST>::ld(in ? Gc + gin_off<FACE, TAB>(p, lk, i) : Gc + i * p.ld);
                g[i] = in ? v : wall_value<FACE>(p, opp7(i), v, th_rd);
            }
        }
        collide(p, f, g);
        if (fast) {
            Store<ST>::st_stream(Fc, f[0]);
#pragma unroll
            for (int i = 1; i < 19; ++i)  // towards an x wall: stays in slot opp(i)
                Store<ST>::st_stream(xwall(-ex(i), xlo, xhi) ? Fc + opp(i) * p.ld : Fc + fout_off<FACE, TAB>(p, lk, i),
                                     f[i]);
            Store<ST>::st_stream(Gc, g[0]);
#pragma unroll
            for (int i = 1; i < 7; ++i)
                Store<ST>::st_stream(xwall(-tx(i), xlo, xhi) ? Gc + opp7(i) * p.ld : Gc + gout_off<FACE, TAB>(p, lk, i),
                                     g[i]);
            return;
        }
        Store<ST>::st_stream(Fc, f[0]);
#pragma unroll
        for (int i = 1; i < 19; ++i)
            Store<ST>::st_stream(((lm >> opp(i)) & 1u) ? Fc + fout_off<FACE, TAB>(p, lk, i) : Fc + opp(i) * p.ld, f[i]);
        if (COND) {
            // x + t_i = x - e_opp(i): inside (bit opp(i) of im) and solid (bit opp(i) of lm clear)
            unsigned other = 0;
#pragma unroll
            for (int i = 1; i < 7; ++i)
                if (((im >> opp7(i)) & 1u) && !((lm >> opp(i)) & 1u)) other |= 1u << i;
            if (other) cross_phase(p, other, a == jsc - 1, spost, col, g);
        }
    } else if (COND) {
        // the solid's own g: pulled as for a liquid node, collided at u = 0
        const unsigned ims = off_walls ? 0x7eu : inside_mask(p, x, y, z);
        const float th_rd = __ldg(thw_rd + col);
        g[0] = Store<ST>::ld(Gc);
#pragma unroll
        for (int i = 1; i < 7; ++i) {
            const bool in = (ims >> i) & 1u;
            const float v = Store<ST>::ld(in ? Gc + gin_off<FACE, TAB>(p, lk, i) : Gc + i * p.ld);
            g[i] = in ? v : wall_value<FACE>(p, opp7(i), v, th_rd);
        }
        collide_solid(p, g);
        if (a <= (nbv & 0xffff)) {
            const unsigned other = other_phase7<FACE>(p, js, x, y, z, false);
            if (other) cross_phase(p, other, a == jsc, gpost, col, g);
        }
    } else {
        if (deep_solid(p, a, nbv)) return;
        solid_post(p, a == jsc, gpost, col, g);
    }
    const unsigned im = off_walls ? 0x7eu : inside_mask(p, x, y, z);
    const float th_wr = __ldg(thw_wr + col);
    Store<ST>::st_stream(Gc, g[0]);
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const bool out = (im >> opp7(i)) & 1u;
        Store<ST>::st_stream(out ? Gc + gout_off<FACE, TAB>(p, lk, i) : Gc + opp7(i) * p.ld,
                      out ? g[i] : wall_value<FACE>(p, i, g[i], th_wr));
    }
}

// The odd step of one node with its loads before step_launch_wait (see
// k_even).  A node that was liquid reads what the flags before the front
// update prescribe (counts js_old, bounds nb_old), which no other thread
// writes, with one exception: the slot it holds towards a node that has just
// become liquid, which that node's thread may have written already.  Those
// links are read again after the wait, from where flip_column moved the
// value.  `inner`: interior under the old flags and, counts changing by at
// most one a step, under the new ones.
template <typename ST, int FACE, bool SNAP>
__device__ __forceinline__ void odd_node_early(const KP &p, const Links *lk, ST *__restrict__ F, ST *__restrict__ G,
                                               const int *js, const int *js_old, const int *nb, const int *nb_old,
                                               const float *gpost, const float *thw_rd,
                                               const float *__restrict__ thw_wr, const int *jmax, int early_blocks,
                                               bool on, int x, int y, int z, const double *s, const SnapOut &snap) {
    const long long c = on ? node_index(p, x, y, z) : 0;
    const int a = axial<FACE>(x, y, z), col = on ? column<FACE>(p, x, y, z) : 0;
    const int q = FACE == 0 ? z : y, nq = FACE == 0 ? p.nz : p.ny;
    const bool off_qa = q >= 1 && q <= nq - 2 && a >= 1 && a <= p.H - 2;
    const bool xlo = x == 0, xhi = x == p.nx - 1;
    unsigned need = 0x7fffeu;  // the links that an interior node has
    if (xlo | xhi) {
#pragma unroll
        for (int i = 1; i < 19; ++i)
            if (xwall(ex(i), xlo, xhi)) need &= ~(1u << i);
    }
    ST *const Fc = F + c;
    ST *const Gc = G + c;
    float f[19], g[7];
    unsigned lm = need, im = 0x7eu;
    bool inner = false, was = false;
    auto pull_g = [&]() {
        const float th_rd = ld_l2(thw_rd + col);
        g[0] = ld_l2(Gc);
#pragma unroll
        for (int i = 1; i < 7; ++i) {
            const bool in = (im >> i) & 1u;
            const float v = ld_l2(in ? Gc + lk->gin[i] : Gc + i * p.ld);
            g[i] = in ? v : wall_value<FACE>(p, opp7(i), v, th_rd);
        }
    };
    const bool late = k1_late(early_blocks);
    if (late) step_launch_wait();
    if (on) {
        const int jm = jmax ? (late ? *jmax : ld_l2(jmax)) : 1 << 29;
        const int jso = late ? js_old[col] : ld_l2(js_old + col);
        const int nbo = late ? nb_old[col] : ld_l2(nb_old + col);
        on = k1_low<FACE>() < jm + 3;
        was = on && a < jso;
        inner = was && off_qa && a + 2 < (nbo >> 16);
        bool fast = inner;
        if (was && !inner) {
            int js9[9];
            load_js9_l2(p, js_old, x, q, js9);
            lm = link_mask9<FACE>(js9, a);
            im = inside_mask(p, x, y, z);
            fast = off_qa && (lm & need) == need;
        }
        if (was && fast) {
#pragma unroll
            for (int i = 0; i < 19; ++i) f[i] = ld_l2(Fc + lk->fin[i]);
#pragma unroll
            for (int i = 0; i < 7; ++i) g[i] = ld_l2(Gc + lk->gin[i]);
            if (xlo | xhi) {  // across an x wall: bounce-back (see odd_node)
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (xwall(ex(i), xlo, xhi)) f[i] = ld_l2(Fc + i * p.ld);
#pragma unroll
                for (int i = 1; i < 7; ++i)
                    if (xwall(tx(i), xlo, xhi)) g[i] = ld_l2(Gc + i * p.ld);
            }
        } else if (was) {
            f[0] = ld_l2(Fc);
#pragma unroll
            for (int i = 1; i < 19; ++i) f[i] = ld_l2(((lm >> i) & 1u) ? Fc + lk->fin[i] : Fc + i * p.ld);
            pull_g();
        }
    }
    if (!late) step_launch_wait();
    if (!on) return;
    const int jsc = inner && !SNAP ? p.H : js[col];
    if (SNAP && a == 0) snap_column(snap, col, s[col], jsc, nb[col]);
    if (a < jsc) {
        bool fast = inner;
        if (!inner) {
            int js9[9];
            load_js9(p, js, x, q, js9);
            const unsigned now = link_mask9<FACE>(js9, a);
            if (!was) {
                im = inside_mask(p, x, y, z);
#pragma unroll
                for (int i = 0; i < 19; ++i) f[i] = 0.0f;
                pull_g();
            } else if (now & ~lm) {
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    if (((now & ~lm) >> i) & 1u) f[i] = ld_l2(Fc + lk->fin[i]);
            }
            lm = now;
            fast = off_qa && (lm & need) == need;
        }
        if (SNAP) snap_node(p, snap, x, y, z, f, g);
        collide(p, f, g);
        Store<ST>::st_stream(Fc, f[0]);
        if (fast) {
#pragma unroll
            for (int i = 1; i < 19; ++i)  // towards an x wall: stays in slot opp(i)
                Store<ST>::st_stream(xwall(-ex(i), xlo, xhi) ? Fc + opp(i) * p.ld : Fc + lk->fout[i], f[i]);
            Store<ST>::st_stream(Gc, g[0]);
#pragma unroll
            for (int i = 1; i < 7; ++i)
                Store<ST>::st_stream(xwall(-tx(i), xlo, xhi) ? Gc + opp7(i) * p.ld : Gc + lk->gout[i], g[i]);
            return;
        }
#pragma unroll
        for (int i = 1; i < 19; ++i)
            Store<ST>::st_stream(((lm >> opp(i)) & 1u) ? Fc + lk->fout[i] : Fc + opp(i) * p.ld, f[i]);
    } else {
        if (deep_solid(p, a, nb[col])) return;
        im = inside_mask(p, x, y, z);
        if (SNAP && a == jsc) snap_ghost<ST, FACE>(p, G, thw_rd, x, y, z, true, snap);
        solid_post(p, a == jsc, gpost, col, g);
    }
    const float th_wr = __ldg(thw_wr + col);
    Store<ST>::st_stream(Gc, g[0]);
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const bool out = (im >> opp7(i)) & 1u;
        Store<ST>::st_stream(out ? Gc + lk->gout[i] : Gc + opp7(i) * p.ld,
                             out ? g[i] : wall_value<FACE>(p, i, g[i], th_wr));
    }
}

template <typename ST, int FACE, bool SNAP>
__global__ void __launch_bounds__(128, SNAP ? 0 : k1_min_blocks<ST>()) k_odd(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                             const int *js, const int *js_old, const int *nb, const int *nb_old,
                                             const float *gpost, const float *thw_rd,
                                             const float *__restrict__ thw_wr, const __grid_constant__ Links lk,
                                             const int *jmax, int early_blocks, const double *s,
                                             const __grid_constant__ SnapOut snap) {
    int x = 0, y = 0, z = 0;
    const bool on = k1_node<FACE>(p, x, y, z);
    odd_node_early<ST, FACE, SNAP>(p, &lk, F, G, js, js_old, nb, nb_old, gpost, thw_rd, thw_wr, jmax, early_blocks, on, x, y, z, s,
                                   snap);
}

// The odd step with heat conduction in the solid (every node updated).
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_odd_cond(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                                  const int *js, const int *js_old,
                                                  const int *nb,
                                                  const float *gpost, const float *__restrict__ thw_rd,
                                                  const float *__restrict__ thw_wr, const __grid_constant__ Links lk,
                                                  const float *spost) {
    step_launch_wait();
    int x, y, z;
    if (k1_node<FACE>(p, x, y, z))
        odd_node<ST, FACE, true, true>(p, &lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x, y, z, spost);
}


// ------------------------------------------- two nodes per thread (FP16)
// With FP16 storage and an even nx, a thread of the stream-collide takes the
// nodes x0 = 2k and x0 + 1 of a row.  Their slots of a direction are
// adjacent and 4-byte aligned (c = index of x0 is even, ld a multiple of 128,
// and a link offset is even unless the link has an x component), so a pair
// of liquid nodes moves its populations as half2 words and collides in
// packed FP32x2 arithmetic (collide2): about half the instructions per node
// of the one-node kernels, whose FP32 arithmetic, not HBM, bounds them with
// 2-byte populations.  A pair that meets the interface (or, in the odd step,
// a wall of the heating axis or of the other in-plane axis) takes the
// one-node code for each of its nodes.
// Resident blocks of 128 the pair kernels ask for (the register budget of a
// thread is 65536 / (128 x this)): 5, 96 registers and under 90 bytes of
// spills, ran the 256^3 FP16 stream-collide in 0.148 ms against 0.158 ms with
// 4 (128 registers, no spills) and 0.164 ms with 6 (80 registers, up to
// 256 bytes of spills).
#ifndef LBM_PAIR_MIN_BLOCKS
#define LBM_PAIR_MIN_BLOCKS 5
#endif
#ifndef LBM_PAIR_MIN_BLOCKS_F32
#define LBM_PAIR_MIN_BLOCKS_F32 5
#endif
template <typename ST> constexpr int pair_min_blocks() {
    return sizeof(ST) == 2 ? LBM_PAIR_MIN_BLOCKS : LBM_PAIR_MIN_BLOCKS_F32;
}

// LIN: 0 rows, 1 columns in a line (known at compile time: with FP16 storage
// the test alone cost spills, 156.5 -> 162 us at 256^3).
template <int FACE, int LIN>
__device__ __forceinline__ bool k1_pair(const KP &p, int &x, int &y, int &z) {
    const int a0 = k1_low<FACE>();
    x = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (LIN) {  // x / nx and x % nx of an even nx: whole pairs
        const int q = (int)((unsigned)x / (unsigned)p.nx);
        x -= q * p.nx;
        y = FACE == 0 ? a0 : q;
        z = FACE == 0 ? q : a0;
        return q < p.P2 && a0 < p.H;
    }
    if (FACE == 0) {
        y = a0 + (int)threadIdx.y;
        z = (int)blockIdx.y;
    } else {
        y = (int)(blockIdx.y * blockDim.y + threadIdx.y);
        z = (int)blockIdx.z;
    }
    return x < p.nx && y < p.ny;
}

// The two adjacent populations of a pair (an aligned half2 or float2 word).
__device__ __forceinline__ float2 ld_pair(const __half *q) { return __half22float2(*(const __half2 *)q); }
__device__ __forceinline__ float2 ld_pair(const float *q) { return *(const float2 *)q; }
__device__ __forceinline__ float2 ld_pair_l2(const float *q) { return ld_l2((const float2 *)q); }
__device__ __forceinline__ float2 ld_pair_l2(const __half *q) {
    unsigned v;
    asm volatile("ld.global.cg.u32 %0, [%1];\n" : "=r"(v) : "l"(q));
    return __half22float2(*(const __half2 *)&v);
}
__device__ __forceinline__ void st_pair(__half *q, float2 v) { __stcs((__half2 *)q, __floats2half2_rn(v.x, v.y)); }
__device__ __forceinline__ void st_pair(float *q, float2 v) { __stcs((float2 *)q, v); }

// The even step of a pair of liquid nodes (both collide, no phase test): its
// loads (EARLY: ones that may stand before step_launch_wait), then the rest.
template <typename ST, typename IX, bool EARLY>
__device__ __forceinline__ void even_pair_load(const KP &p, const ST *F, const ST *G, IX c, float2 (&f)[19],
                                               float2 (&g)[7]) {
#pragma unroll
    for (int i = 0; i < 19; ++i)
        f[i] = EARLY ? ld_pair_l2(elem<IX>(F, c, i * p.ld)) : ld_pair(elem<IX>(F, c, i * p.ld));
#pragma unroll
    for (int i = 0; i < 7; ++i)
        g[i] = EARLY ? ld_pair_l2(elem<IX>(G, c, i * p.ld)) : ld_pair(elem<IX>(G, c, i * p.ld));
}
template <typename ST, typename IX>
__device__ __forceinline__ void even_pair_finish(const KP &p, ST *__restrict__ F, ST *__restrict__ G, IX c,
                                                 float2 (&f)[19], float2 (&g)[7]) {
    collide2<sizeof(ST) == 4>(p, f, g);
#pragma unroll
    for (int i = 0; i < 19; ++i) st_pair(elem<IX>(F, c, opp(i) * p.ld), f[i]);
#pragma unroll
    for (int i = 0; i < 7; ++i) st_pair(elem<IX>(G, c, opp7(i) * p.ld), g[i]);
}
template <typename ST, typename IX>
__device__ __forceinline__ void even_pair_liquid(const KP &p, ST *__restrict__ F, ST *__restrict__ G, IX c) {
    float2 f[19], g[7];
    even_pair_load<ST, IX, false>(p, F, G, c, f, g);
    even_pair_finish<ST, IX>(p, F, G, c, f, g);
}

template <typename ST, int FACE, typename IX>
__device__ __forceinline__ void even_pair(const KP &p, ST *__restrict__ F, ST *__restrict__ G,
                                          const int *js, const int *nb,
                                          const float *gpost, int x, int y, int z) {
    const int a = axial<FACE>(x, y, z);
    const int col = column<FACE>(p, x, y, z);  // x + 1 is in column col + 1
    if (a < js[col] && a < js[col + 1]) {
        even_pair_liquid<ST, IX>(p, F, G, (IX)node_index(p, x, y, z));
    } else {
        even_node<ST, FACE, IX>(p, F, G, js, nb, gpost, x, y, z);
        even_node<ST, FACE, IX>(p, F, G, js, nb, gpost, x + 1, y, z);
    }
}

template <typename ST, int FACE, typename IX, int LIN>
__global__ void __launch_bounds__(128, pair_min_blocks<ST>()) k_even_pair(const __grid_constant__ KP p, ST *__restrict__ F,
                                                      ST *__restrict__ G, const int *js,
                                                      const int *nb, const float *gpost,
                                                      const int *jmax) {
    step_launch_wait();
    int x, y, z;
    if (k1_pair<FACE, LIN>(p, x, y, z) && !(jmax && k1_low<FACE>() >= *jmax + 3)) even_pair<ST, FACE, IX>(p, F, G, js, nb, gpost, x, y, z);
}

// The odd step of a pair on the fast path (both liquid, off the walls of the
// heating axis and of the other in-plane axis, every link streaming but
// those across an x wall).  Links without an x component move as half2 /
// float2 words; the others node by node, with the x walls (x0 = 0 for lane
// x, x0 + 1 = nx - 1 for lane y) taken as in odd_node.
template <typename ST, int FACE, typename IX, bool EARLY>
__device__ __forceinline__ void odd_pair_load(const KP &p, const Links *lk, const ST *F, const ST *G, int x, int y,
                                              int z, float2 (&f)[19], float2 (&g)[7]) {
    const IX c = (IX)node_index(p, x, y, z), c1 = c + 1;
    const bool xlo = x == 0, xhi = x + 1 == p.nx - 1;
    auto one = [](const ST *q) { return EARLY ? ld_l2(q) : Store<ST>::ld(q); };
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        if (ex(i) == 0) {
            f[i] = EARLY ? ld_pair_l2(elem<IX>(F, c, lk->fin[i])) : ld_pair(elem<IX>(F, c, lk->fin[i]));
        } else {
            // across an x wall: bounce-back from the node's own slot i
            f[i].x = one(elem<IX>(F, c, ex(i) > 0 && xlo ? i * p.ld : lk->fin[i]));
            f[i].y = one(elem<IX>(F, c1, ex(i) < 0 && xhi ? i * p.ld : lk->fin[i]));
        }
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        if (tx(i) == 0) {
            g[i] = EARLY ? ld_pair_l2(elem<IX>(G, c, lk->gin[i])) : ld_pair(elem<IX>(G, c, lk->gin[i]));
        } else {
            g[i].x = one(elem<IX>(G, c, tx(i) > 0 && xlo ? i * p.ld : lk->gin[i]));
            g[i].y = one(elem<IX>(G, c1, tx(i) < 0 && xhi ? i * p.ld : lk->gin[i]));
        }
    }
}
template <typename ST, int FACE, typename IX>
__device__ __forceinline__ void odd_pair_finish(const KP &p, const Links *lk, ST *__restrict__ F, ST *__restrict__ G,
                                                int x, int y, int z, float2 (&f)[19], float2 (&g)[7]) {
    const IX c = (IX)node_index(p, x, y, z), c1 = c + 1;
    const bool xlo = x == 0, xhi = x + 1 == p.nx - 1;
    collide2<sizeof(ST) == 4>(p, f, g);
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        if (ex(i) == 0) {
            st_pair(elem<IX>(F, c, lk->fout[i]), f[i]);
        } else {
            // towards an x wall: stays in the node's slot opp(i)
            Store<ST>::st_stream(elem<IX>(F, c, ex(i) < 0 && xlo ? opp(i) * p.ld : lk->fout[i]), f[i].x);
            Store<ST>::st_stream(elem<IX>(F, c1, ex(i) > 0 && xhi ? opp(i) * p.ld : lk->fout[i]), f[i].y);
        }
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        if (tx(i) == 0) {
            st_pair(elem<IX>(G, c, lk->gout[i]), g[i]);
        } else {
            Store<ST>::st_stream(elem<IX>(G, c, tx(i) < 0 && xlo ? opp7(i) * p.ld : lk->gout[i]), g[i].x);
            Store<ST>::st_stream(elem<IX>(G, c1, tx(i) > 0 && xhi ? opp7(i) * p.ld : lk->gout[i]), g[i].y);
        }
    }
}
template <typename ST, int FACE, typename IX>
__device__ __forceinline__ void odd_pair_liquid(const KP &p, const Links *lk, ST *__restrict__ F, ST *__restrict__ G,
                                                int x, int y, int z) {
    float2 f[19], g[7];
    odd_pair_load<ST, FACE, IX, false>(p, lk, F, G, x, y, z, f, g);
    odd_pair_finish<ST, FACE, IX>(p, lk, F, G, x, y, z, f, g);
}

// The odd step for a pair: both nodes on the one-node fast path (liquid, off
// the walls of the heating axis and of the other in-plane axis, one node
// below the lowest first-solid node of their 3x3 columns) take
// odd_pair_liquid, any other pair the one-node code node by node.
template <typename ST, int FACE, typename IX>
__device__ __forceinline__ void odd_pair(const KP &p, const Links *lk, ST *__restrict__ F,
                                         ST *__restrict__ G, const int *js,
                                         const int *js_old, const int *nb,
                                         const float *gpost, const float *__restrict__ thw_rd,
                                         const float *__restrict__ thw_wr, int x, int y, int z) {
    const int a = axial<FACE>(x, y, z);
    const int col = column<FACE>(p, x, y, z);
    const int q = FACE == 0 ? z : y, nq = FACE == 0 ? p.nz : p.ny;
    const bool off_qa = q >= 1 && q <= nq - 2 && a >= 1 && a <= p.H - 2;
    const int b0 = nb[col] >> 16, b1 = nb[col + 1] >> 16;
    if (!(off_qa && a + 1 < b0 && a + 1 < b1)) {
        int c12[12], js9[9], mn, mx;
        load_js12(p, js, x, q, c12);
        range_js12(p, c12, x, q, mn, mx);
        if (!(off_qa && a + 1 < mn)) {  // the bounds may be two low
            js9_of_js12(c12, 0, js9);
            odd_node<ST, FACE>(p, lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x, y, z, nullptr, js9);
            js9_of_js12(c12, 1, js9);
            odd_node<ST, FACE>(p, lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x + 1, y, z, nullptr, js9);
            return;
        }
    }
    odd_pair_liquid<ST, FACE, IX>(p, lk, F, G, x, y, z);
}

template <typename ST, int FACE, typename IX, int LIN>
__global__ void __launch_bounds__(128, pair_min_blocks<ST>()) k_odd_pair(const __grid_constant__ KP p, ST *__restrict__ F,
                                                     ST *__restrict__ G, const int *js,
                                                     const int *js_old, const int *nb,
                                                     const float *gpost,
                                                     const float *__restrict__ thw_rd,
                                                     const float *__restrict__ thw_wr,
                                                     const __grid_constant__ Links lk, const int *jmax) {
    step_launch_wait();
    int x, y, z;
    if (k1_pair<FACE, LIN>(p, x, y, z) && !(jmax && k1_low<FACE>() >= *jmax + 3)) odd_pair<ST, FACE, IX>(p, &lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x, y, z);
}


// The pair kernels of the middle sizes (FP32 storage, up to 160^3 nodes): the
// first wave's pairs load before step_launch_wait, like the one-node kernels
// (k_even, k_odd): the even step's pairs that were liquid before the front
// update, the odd step's that are interior whatever it does.  128^3 with a
// thin layer 15.5 -> 14.4 us a step (16.5 with one node per thread), at 0.45 H
// 39.8 -> 37.6 (40.4).  Larger grids take the plain kernels: a first wave is
// little of them (256^3 FP32 the same), and with FP16 storage the second set
// of loads cost more than it hid (156.5 -> 161.7 us).
// SNAP: see k_even; a pair that is split takes its snapshot by gathers, from
// the slots that its nodes own in this step.
template <typename ST, int FACE, typename IX, int LIN, bool SNAP>
__global__ void __launch_bounds__(128, pair_min_blocks<ST>()) k_even_pair_early(const __grid_constant__ KP p, ST *__restrict__ F,
                                                      ST *__restrict__ G, const int *js, const int *js_old,
                                                      const int *nb, const float *gpost,
                                                      const int *jmax, int early_blocks, const double *s,
                                                      const __grid_constant__ SnapOut snap) {
    int x = 0, y = 0, z = 0;
    const bool on = k1_pair<FACE, LIN>(p, x, y, z), late = k1_late(early_blocks);
    if (late) step_launch_wait();
    const IX c = on ? (IX)node_index(p, x, y, z) : 0;
    const int a = axial<FACE>(x, y, z);
    const int col = on ? column<FACE>(p, x, y, z) : 0;  // x + 1 is in column col + 1
    float2 f[19], g[7];
    bool low = true, loaded = false;
    if (late) {
        low = !jmax || k1_low<FACE>() < *jmax + 3;
    } else {
        const int jm = jmax ? ld_l2(jmax) : 1 << 29;
        const int2 jo = ld_l2((const int2 *)(js_old + col));
        low = k1_low<FACE>() < jm + 3;
        loaded = on && low && a < jo.x && a < jo.y;
        if (loaded) even_pair_load<ST, IX, true>(p, F, G, c, f, g);
        step_launch_wait();
    }
    if (!on || !low) return;
    if (SNAP && a == 0) snap_pair_columns(snap, col, s, js, nb);
    if (!(a < js[col] && a < js[col + 1])) {
        if (SNAP) {
            snap_any<ST, FACE>(p, F, G, js, js_old, nullptr, x, y, z, false, snap);
            snap_any<ST, FACE>(p, F, G, js, js_old, nullptr, x + 1, y, z, false, snap);
        }
        even_node<ST, FACE, IX>(p, F, G, js, nb, gpost, x, y, z);
        even_node<ST, FACE, IX>(p, F, G, js, nb, gpost, x + 1, y, z);
        return;
    }
    if (!loaded) even_pair_load<ST, IX, false>(p, F, G, c, f, g);
    if (SNAP) snap_pair(p, snap, x, y, z, f, g);
    even_pair_finish<ST, IX>(p, F, G, c, f, g);
}

template <typename ST, int FACE, typename IX, int LIN, bool SNAP>
__global__ void __launch_bounds__(128, pair_min_blocks<ST>()) k_odd_pair_early(const __grid_constant__ KP p, ST *__restrict__ F,
                                                     ST *__restrict__ G, const int *js, const int *js_old,
                                                     const int *nb, const int *nb_old,
                                                     const float *gpost,
                                                     const float *__restrict__ thw_rd,
                                                     const float *__restrict__ thw_wr,
                                                     const __grid_constant__ Links lk, const int *jmax,
                                                     int early_blocks, const double *s,
                                                     const __grid_constant__ SnapOut snap) {
    int x = 0, y = 0, z = 0;
    const bool on = k1_pair<FACE, LIN>(p, x, y, z), late = k1_late(early_blocks);
    if (late) step_launch_wait();
    const int a = axial<FACE>(x, y, z);
    const int col = on ? column<FACE>(p, x, y, z) : 0;
    const int q = FACE == 0 ? z : y, nq = FACE == 0 ? p.nz : p.ny;
    const bool off_qa = q >= 1 && q <= nq - 2 && a >= 1 && a <= p.H - 2;
    float2 f[19], g[7];
    bool low = true, loaded = false;
    if (late) {
        low = !jmax || k1_low<FACE>() < *jmax + 3;
    } else {
        const int jm = jmax ? ld_l2(jmax) : 1 << 29;
        const int2 bo = ld_l2((const int2 *)(nb_old + col));
        low = k1_low<FACE>() < jm + 3;
        // interior under the counts before the front update less one, so under the new ones
        loaded = on && low && off_qa && a + 2 < (bo.x >> 16) && a + 2 < (bo.y >> 16);
        if (loaded) odd_pair_load<ST, FACE, IX, true>(p, &lk, F, G, x, y, z, f, g);
        step_launch_wait();
    }
    if (!on || !low) return;
    if (SNAP && a == 0) snap_pair_columns(snap, col, s, js, nb);
    if (!loaded) {
        const int b0 = nb[col] >> 16, b1 = nb[col + 1] >> 16;
        if (!(off_qa && a + 1 < b0 && a + 1 < b1)) {
            int c12[12], js9[9], mn, mx;
            load_js12(p, js, x, q, c12);
            range_js12(p, c12, x, q, mn, mx);
            if (!(off_qa && a + 1 < mn)) {  // the bounds may be two low
                if (SNAP) {
                    snap_any<ST, FACE>(p, F, G, js, js_old, thw_rd, x, y, z, true, snap);
                    snap_any<ST, FACE>(p, F, G, js, js_old, thw_rd, x + 1, y, z, true, snap);
                }
                js9_of_js12(c12, 0, js9);
                odd_node<ST, FACE>(p, &lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x, y, z, nullptr, js9);
                js9_of_js12(c12, 1, js9);
                odd_node<ST, FACE>(p, &lk, F, G, js, js_old, nb, gpost, thw_rd, thw_wr, x + 1, y, z, nullptr, js9);
                return;
            }
        }
        odd_pair_load<ST, FACE, IX, false>(p, &lk, F, G, x, y, z, f, g);
    }
    if (SNAP) snap_pair(p, snap, x, y, z, f, g);
    odd_pair_finish<ST, FACE, IX>(p, &lk, F, G, x, y, z, f, g);
}


// -------------------------------------------------- state gathers (natural)
// Shifted pre-collision g of node (x,y,z).  In flight: pull from the
// neighbours' slots (walls by their rules with wall field thw); natural:
// the node's own slots.
// One branch for the layout and addresses chosen by selects: with a branch per
// direction every load waited for the one before it (its conversion to FP32
// with FP16 storage above all: the fields of a 256^3 FP16 state took 441 us to
// read, now 190, its distributions 527, now 355; in flight 490, now 228).
template <typename ST, int FACE>
__device__ __forceinline__ void gather_g(const KP &p, const ST *G, int x, int y, int z, bool inflight,
                                         const float *thw, float (&g)[7]) {
    const ST *Gc = G + node_index(p, x, y, z);
    if (!inflight) {
#pragma unroll
        for (int i = 0; i < 7; ++i) g[i] = Store<ST>::ld(Gc + i * p.ld);
        return;
    }
    const unsigned im = inside_mask(p, x, y, z);
    const float Tw = axial<FACE>(x, y, z) == 0 ? thw[column<FACE>(p, x, y, z)] : 0.0f;
    g[0] = Store<ST>::ld(Gc);
#pragma unroll
    for (int i = 1; i < 7; ++i)
        g[i] = Store<ST>::ld(((im >> i) & 1u) ? Gc + (opp7(i) * p.ld - off7<FACE>(p, i)) : Gc + i * p.ld);
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const int w = wall_of_link<FACE>(opp7(i));
        if (w != 3 && !((im >> i) & 1u)) g[i] = -g[i] + 2.0f * w7(i) * ((w == 1 ? Tw : p.Tc) - p.Ts);
    }
}

template <typename ST, int FACE>
__device__ __forceinline__ void snap_ghost(const KP &p, const ST *G, const float *thw, int x, int y, int z,
                                           bool inflight, const SnapOut &o) {
    if (axial<FACE>(x, y, z) >= o.heights) return;
    float f[19], g[7];
    gather_g<ST, FACE>(p, G, x, y, z, inflight, thw, g);
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = 0.0f;
    snap_node(p, o, x, y, z, f, g);
}

// Shifted pre-collision f of a liquid node.  js: the liquid flags that the
// in-flight values were produced under, or the ones after flip_column has run.
template <typename ST, int FACE, bool FIXED = false>
__device__ __forceinline__ void gather_f(const KP &p, const ST *F, const int *js, int x, int y, int z,
                                         bool inflight, float (&f)[19]) {
    const ST *Fc = F + node_index(p, x, y, z);
    if (!inflight) {
#pragma unroll
        for (int i = 0; i < 19; ++i) f[i] = Store<ST>::ld(Fc + i * p.ld);
        return;
    }
    int js9[9];
    load_js9<FIXED>(p, js, x, FACE == 0 ? z : y, js9);
    const unsigned lm = link_mask9<FACE>(js9, axial<FACE>(x, y, z));
    f[0] = Store<ST>::ld(Fc);
#pragma unroll
    for (int i = 1; i < 19; ++i)
        f[i] = Store<ST>::ld(((lm >> i) & 1u) ? Fc + (opp(i) * p.ld - off19<FACE>(p, i)) : Fc + i * p.ld);
}

// gather_f of the state between steps (flip_column has run): a node that has
// become liquid since the in-flight values were produced (under js_old)
// starts from fh = 0 (in the natural layout its slots hold that).  FIXED: see
// load_js9.
template <typename ST, int FACE, bool FIXED = true>
__device__ __forceinline__ void gather_f_now(const KP &p, const ST *F, const int *js, const int *js_old, int x, int y,
                                             int z, bool inflight, float (&f)[19]) {
    if (inflight && axial<FACE>(x, y, z) >= js_old[column<FACE>(p, x, y, z)]) {
#pragma unroll
        for (int i = 0; i < 19; ++i) f[i] = 0.0f;
        return;
    }
    gather_f<ST, FACE, FIXED>(p, F, js, x, y, z, inflight, f);
}

template <typename ST, int FACE>
__device__ __forceinline__ void snap_any(const KP &p, const ST *F, const ST *G, const int *js, const int *js_old,
                                         const float *thw, int x, int y, int z, bool inflight, const SnapOut &o) {
    const int a = axial<FACE>(x, y, z), jsc = js[column<FACE>(p, x, y, z)];
    if (a > jsc) return;
    if (a == jsc) {
        snap_ghost<ST, FACE>(p, G, thw, x, y, z, inflight, o);
        return;
    }
    float f[19], g[7];
    gather_g<ST, FACE>(p, G, x, y, z, inflight, thw, g);
    gather_f_now<ST, FACE, false>(p, F, js, js_old, x, y, z, inflight, f);
    snap_node(p, o, x, y, z, f, g);
}

// gather_f in flight for the node at height a of the middle column, with
// the liquid tests read from js9 (load_js9) instead of memory.
template <typename ST, int FACE>
__device__ __forceinline__ void gather_f9(const KP &p, const ST *F, const int (&js9)[9], int x, int y, int z, int a,
                                          float (&f)[19]) {
    const ST *Fc = F + node_index(p, x, y, z);
    const unsigned lm = link_mask9<FACE>(js9, a);
    f[0] = Store<ST>::ld(Fc);
#pragma unroll
    for (int i = 1; i < 19; ++i)
        f[i] = Store<ST>::ld(((lm >> i) & 1u) ? Fc + (opp(i) * p.ld - off19<FACE>(p, i)) : Fc + i * p.ld);
}

// Ts + the sum of the shifted g (the temperature the front reads; FP32, the
// precision the populations are held in).
__device__ __forceinline__ float sum_T(const KP &p, const float (&g)[7]) {
    float t = 0.0f;
#pragma unroll
    for (int i = 0; i < 7; ++i) t += g[i];
    return p.Ts + t;
}

template <typename ST, int FACE>
__device__ __forceinline__ float node_T(const KP &p, const ST *G, int col, int j, bool inflight, const float *thw) {
    int x, y, z;
    column_node<FACE>(p, col, j, x, y, z);
    float g[7];
    gather_g<ST, FACE>(p, G, x, y, z, inflight, thw, g);
    return sum_T(p, g);
}

// Where a front height s lies: n = floor(s) held to [-1, H], and fr = s - n
// (exact; in [0, 1) for a front inside the cavity).  Every distance from s to
// a node centre is then one exact FP64 addition of a constant to fr.  FP64
// issues at a small fraction of the FP32 rate here (about two lanes an SM and
// clock), and the front update spent up to forty FP64 operations and
// conversions a column on node centres made from integers; this form has
// about twenty, with the same values.
struct FrontPos {
    int n;
    double fr;
};
__device__ __forceinline__ FrontPos front_pos(double s, int H) {
    FrontPos f;
    f.n = __double2int_rd(s);  // saturates; NaN: a value below -1
    f.n = f.n > H ? H : (f.n < -1 ? -1 : f.n);
    f.fr = s - (double)f.n;
    return f;
}
// Highest node at least half a cell below the front (centre j + 1/2 <= s -
// 1/2), or -1.
__device__ __forceinline__ int guarded_node(const FrontPos &f) { return f.n >= 1 ? f.n - 1 : -1; }
// s minus the centre of that node, and of the one below it.
__device__ __forceinline__ float guarded_distance(const FrontPos &f) { return (float)(f.fr + 0.5); }
__device__ __forceinline__ float below_distance(const FrontPos &f) { return (float)(f.fr + 1.5); }
// Liquid nodes of the column: j + 1/2 < s, i.e. ceil(s - 1/2), within [0, H].
__device__ __forceinline__ int liquid_count(const FrontPos &f, int H) {
    const int j = f.n + (f.fr > 0.5 ? 1 : 0);
    return j < 0 ? 0 : (j > H ? H : j);
}
// Whether a new front has left [1/2, H] (NaN has): the bounds are looked at
// only where floor(s) is next to them.
__device__ __forceinline__ bool front_clamped(double s, const FrontPos &f, int H) {
    return f.n >= H ? s > (double)H : (f.n < 1 && !(s >= 0.5));
}
// Centre of the first solid node jn minus s (jn from liquid_count, below H).
__device__ __forceinline__ float ghost_distance(const FrontPos &f, int jn) {
    return (float)((jn == f.n ? 0.5 : 1.5) - f.fr);
}

// The Eq. 6 gradient dT/da at the front a = s (R8: the one-sided quadratic
// through (s, Tm) and the guarded node k with the node below it, or the
// heated wall (0, Tw) for a missing node; linear through the wall when k <
// 0), and the front speed ds/dt = coef (1 + s_p^2 + s_q^2)(-dT/da).  FP32
// with every operation rounded on its own (no contraction into FMAs), so that
// each kernel that evaluates them (the front update, the ensemble, the
// adjoint's recomputation) gets the same bits.  With h = x1 - x0,
// d1 = s - x1, d0 = s - x0: p'(s) = (y0 d1^2 - y1 d0^2 + Tm h (d0 + d1)) /
// (h d0 d1).
__device__ __forceinline__ float front_gradient(int k, double sc, const FrontPos &f, float y0, float y1, float Tm,
                                                float Tw) {
    if (k < 0) return __fdiv_rn(__fsub_rn(Tm, Tw), (float)sc);
    const float h = k >= 1 ? 1.0f : 0.5f;
    const float d1 = guarded_distance(f), d0 = k >= 1 ? below_distance(f) : (float)sc;
    const float num = __fadd_rn(__fsub_rn(__fmul_rn(__fmul_rn(y0, d1), d1), __fmul_rn(__fmul_rn(y1, d0), d0)),
                                __fmul_rn(__fmul_rn(Tm, h), __fadd_rn(d0, d1)));
    return __fdiv_rn(num, __fmul_rn(__fmul_rn(h, d0), d1));
}
__device__ __forceinline__ float front_slope_factor(float sp, float sq) {
    return __fadd_rn(__fadd_rn(1.0f, __fmul_rn(sp, sp)), __fmul_rn(sq, sq));
}
__device__ __forceinline__ float front_speed(const KP &p, float fac, float G) {
    return __fmul_rn(__fmul_rn(p.coef_f, fac), -G);
}

// Lowest node at least half a cell above s (centre j + 1/2 >= s + 1/2, i.e.
// j = ceil(s)), or H when there is none.
__device__ __forceinline__ int guarded_solid_node(double s, int H) {
    const int k = (int)ceil(s);
    return k > H ? H : k;
}

// Solid-side dT/da at the front a = s (the k_s dT_s/da term of Eq. 6, heat
// conduction in the solid): the mirror of front_gradient, the one-sided
// quadratic through (s, Tm), the guarded solid node ks and the node above
// it, the cold wall (H, Tc) standing in for a missing node; linear through
// (s, Tm) and (H, Tc) when ks = H.  Y1, Y2: the temperatures of nodes ks and
// ks + 1 (or the wall) minus Tm, so that a solid at Tm gives exactly zero.
__device__ __forceinline__ float solid_gradient(int ks, int H, double sc, float Y1, float Y2, float Tm, float Tc) {
    if (ks >= H) return (Tc - Tm) / (float)((double)H - sc);
    const double x1 = ks + 0.5, x2 = ks + 1 < H ? ks + 1.5 : (double)H;
    return Y1 * (float)(sc - x2) / ((float)(x1 - sc) * (float)(x1 - x2)) +
           Y2 * (float)(sc - x1) / ((float)(x2 - sc) * (float)(x2 - x1));
}

// Bounds of the liquid counts of the 3x3 columns after a front update, from
// the counts js9 before it (a count changes by at most one a step: a front
// that moves half a node or more is reported as unstable), packed as
// min << 16 | max.  The stream-collide's interior and deep-solid tests use
// them: a bound one node wide of the true one sends a node to the general
// path or updates a node at rest, with the same results.
__device__ __forceinline__ int count_bounds(const KP &p, const int (&js9)[9], int pp, int q) {
    int mn = 1 << 15, mx = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int dp = k % 3 - 1, dq = k / 3 - 1;
        const bool in = (unsigned)(pp + dp) < (unsigned)p.P1 && (unsigned)(q + dq) < (unsigned)p.P2;
        mn = in && js9[k] < mn ? js9[k] : mn;
        mx = js9[k] > mx ? js9[k] : mx;
    }
    return ((mn > 0 ? mn - 1 : 0) << 16) | (mx + 1);
}

// ------------------------------------------------------------------ flip
// Nodes of a column between the old and the new liquid counts (jo, jn)
// changed phase.
// Natural layout: a newly liquid node y gets fh = 0 (f = f^eq(1, 0)).
// In flight, for every node x = y + e_i that was liquid (liquid counts js):
//   y newly liquid: x's population towards y bounced back under the old flags,
//     so it waits in x's own slot i; the odd step, seeing y liquid, looks in
//     slot opp(i) of y, so it is moved there (y's own fh = 0 is left to the
//     readers: see odd_node, gather_f_now);
//   y newly solid: x's population from y waits in slot opp(i) of y; the odd
//     step, seeing y solid, looks in x's own slot i.
// The column's own thread does this right after its front update, while other
// columns are still reading f for their ghosts: no slot written here is one
// that they read.  The first kind writes only slots of a node that was solid,
// and the ghost of a column reads slots of nodes that were liquid; the second
// writes slot i of x, which only the ghost whose source node is y reads, and
// that is this column's, whose source has moved below y.  Flags of the new
// state are not needed: a value moved for a node x that turns solid itself is
// read by nothing.
template <typename ST, int FACE>
__device__ __forceinline__ void flip_column(const KP &p, ST *__restrict__ F, const int *js, bool inflight,
                                            int col, int jo, int jn) {
    const int lo = jo < jn ? jo : jn, hi = jo < jn ? jn : jo;
    for (int j = lo; j < hi; ++j) {
        int x, y, z;
        column_node<FACE>(p, col, j, x, y, z);
        const long long c = node_index(p, x, y, z);
        if (!inflight) {
            if (jo < jn) {
#pragma unroll
                for (int i = 0; i < 19; ++i) Store<ST>::st(F + i * p.ld + c, 0.0f);
            }
            continue;
        }
        // every load before the first store (the compiler cannot move a load
        // above a store into the same array)
        bool on[19];
        float v[19];
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            on[i] = liquid_at<FACE>(p, js, x + ex(i), y + ey(i), z + ez(i));
            const ST *from = jo < jn ? F + i * p.ld + (c + off19<FACE>(p, i)) : F + opp(i) * p.ld + c;
            v[i] = on[i] ? Store<ST>::ld(from) : 0.0f;
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            ST *to = jo < jn ? F + opp(i) * p.ld + c : F + i * p.ld + (c + off19<FACE>(p, i));
            if (on[i]) Store<ST>::st(to, v[i]);
        }
    }
}

// ------------------------------------------------------------ front (Eq. 6)
// One thread per column.  From the state after a step (T of the liquid at
// t + 1, front s_t): the one-sided quadratic gradient at the front, the
// in-plane slopes from the old fronts of the neighbour columns (mirror at
// the side walls), ds/dt = coef (1 + s_p^2 + s_q^2)(-dT/da), the new front
// clamped to [1/2, H], its liquid-node count, and the ghost node of the new
// front: g*_ghost = g^eq(T_ghost, 0) + (g*_L - g^eq(T_L, u_L)).
// move = 0 keeps the front (used to prepare the ghost after a state upload).
// SPEC (as a kernel of its own): wait for the stream-collide once the column's
// own data are loaded, load the ghost's likely source node together with the gradient
// stencil (two dependent load stages instead of three; more registers), and
// flip the column's nodes; without it the caller flips them.
//
// Precision: the front heights are accumulated in FP64 (s + ds, and the
// distances from s to the stencil nodes and the ghost are FP64 differences);
// the gradient, the speed and the ghost temperature are FP32 arithmetic, the
// precision of the temperatures they are made of.  GB300 issues FP64 at a
// small fraction of its FP32 rate, and the FP64 divisions of an all-FP64
// version made this kernel FP64-pipe bound.
//
// COND (heat conduction in the solid): Eq. 6 gains kappa dT_s/da from
// solid_gradient at s_t, and the solid side's ghost populations of the new
// front are written to spost: at the last liquid node, g^eq(T_sghost, 0)
// plus the non-equilibrium part of the first solid node collided at u = 0,
// with T_sghost on the line through (s, Tm) and the guarded solid node (or
// the cold wall); the rest state at Tm in a column without both phases.
template <typename ST, int FACE, bool SPEC = true, bool COND = false>
__device__ __forceinline__ int front_column(const KP &p, ST *__restrict__ F, const ST *G,
                                           const int *__restrict__ js, int *__restrict__ js_next,
                                           int *__restrict__ nb_next, const double *__restrict__ s, double *__restrict__ s_next,
                                           float *__restrict__ gpost, const float *__restrict__ thw, int inflight,
                                           int move, int *__restrict__ status, int col,
                                           float *__restrict__ spost = nullptr) {
    const int P1 = p.P1, P2 = p.P2, H = p.H;
    const int pp = col % P1, q = col / P1;
    const bool infl = inflight != 0;
    // Load stage 1: what depends on the column only.  None of it is written
    // by the stream-collide, so with SPEC it stands before the wait for it.
    const double sc = ld_l2(s + col);
    const float Tm = p.Tm;
    const float Tw = ld_l2(thw + col);
    int js9[9];
    load_js9_l2(p, js, pp, q, js9);
    const int jsc = js9[4];
    float sp = 0.0f, sq = 0.0f;
    if (move) {
        const double sp_hi = ld_l2(s + q * P1 + (pp + 1 < P1 ? pp + 1 : pp)), sp_lo = ld_l2(s + q * P1 + (pp > 0 ? pp - 1 : pp));
        const double sq_hi = ld_l2(s + (q + 1 < P2 ? q + 1 : q) * P1 + pp), sq_lo = ld_l2(s + (q > 0 ? q - 1 : q) * P1 + pp);
        sp = 0.5f * (float)(sp_hi - sp_lo);
        sq = 0.5f * (float)(sq_hi - sq_lo);
    }
    if (SPEC) step_launch_wait();
    nb_next[col] = count_bounds(p, js9, pp, q);
    // Load stage 2: the gradient stencil of s_t and, speculatively, the node
    // below the current front, which is the ghost's source node whenever the
    // liquid count does not change (all but a few columns per step).
    const FrontPos fc = front_pos(sc, H);
    const int k = move ? guarded_node(fc) : -2;
    float y1 = 0.0f, y0 = Tw;
    if (k >= 0) {
        y1 = node_T<ST, FACE>(p, G, col, k, infl, thw);
        if (k >= 1) y0 = node_T<ST, FACE>(p, G, col, k - 1, infl, thw);
    }
    const int L = jsc - 1;
    const bool spec = SPEC && L >= 0 && jsc < H;
    float gL[7], fL[19];
    if (spec) {
        int x, y, z;
        column_node<FACE>(p, col, L, x, y, z);
        gather_g<ST, FACE>(p, G, x, y, z, infl, thw, gL);
        if (infl) gather_f9<ST, FACE>(p, F, js9, x, y, z, L, fL);
        else gather_f<ST, FACE, SPEC>(p, F, js, x, y, z, false, fL);
    }
    // The solid side of the front (conduction in the solid, a column with a
    // solid node): temperatures of the guarded solid node and the one above.
    int ks = H;
    float Ts1 = Tm, Ts2 = Tm, Gs = 0.0f;
    if (COND && move && jsc < H) {
        ks = guarded_solid_node(sc, H);
        if (ks < H) {
            Ts1 = node_T<ST, FACE>(p, G, col, ks, infl, thw);
            Ts2 = ks + 1 < H ? node_T<ST, FACE>(p, G, col, ks + 1, infl, thw) : p.Tc;
        }
        Gs = p.kappa * solid_gradient(ks, H, sc, Ts1 - Tm, Ts2 - Tm, Tm, p.Tc);
    }
    // Then Eq. 6.
    double sn = sc;
    FrontPos fn = fc;
    if (move) {
        const float Gr = front_gradient(k, sc, fc, y0, y1, Tm, Tw);
        const float v = front_speed(p, front_slope_factor(sp, sq), COND ? Gr - Gs : Gr);
        if (!isfinite(Gr) || (COND && !isfinite(Gs))) atomicOr_system(status, 2);
        else if (!(fabsf(v) <= 0.5f)) atomicOr_system(status, 1);
        sn = sc + (double)v;
        fn = front_pos(sn, H);
        if (front_clamped(sn, fn, H)) {
            sn = fn.n >= H ? (double)H : 0.5;
            fn = front_pos(sn, H);
        }
    }
    s_next[col] = sn;
    const int jn = liquid_count(fn, H);
    js_next[col] = jn;
    if (COND) {
        // the solid side's ghost populations at the last liquid node jn - 1
        float sg[7];
        if (jn >= 1 && jn < H) {
            const double yg = jn - 0.5;
            const int ks2 = guarded_solid_node(sn, H);
            float Tsg;
            if (ks2 >= H) {
                Tsg = Tm + (p.Tc - Tm) * (float)((yg - sn) / ((double)H - sn));
            } else {
                float Tk;
                if (move && jsc < H && ks2 == ks) Tk = Ts1;
                else if (move && jsc < H && ks2 == ks + 1 && ks + 1 < H) Tk = Ts2;
                else Tk = node_T<ST, FACE>(p, G, col, ks2, infl, thw);
                Tsg = Tm + (Tk - Tm) * (float)((yg - sn) / ((ks2 + 0.5) - sn));
            }
            float gS[7];
            int x, y, z;
            column_node<FACE>(p, col, jn, x, y, z);
            gather_g<ST, FACE>(p, G, x, y, z, infl, thw, gS);
            const float Th = gS[0] + gS[1] + gS[2] + gS[3] + gS[4] + gS[5] + gS[6];
            const float dTg = Tsg - p.Ts;
#pragma unroll
            for (int i = 0; i < 7; ++i) sg[i] = w7(i) * dTg;
            // N^-1 (I - Q)(n - n^eq) of the solid node at u = 0
            constexpr float i1 = 1.0f / (float)nnorm(1), i4 = 1.0f / (float)nnorm(4);
            constexpr float i5 = 1.0f / (float)nnorm(5), i6 = 1.0f / (float)nnorm(6);
            const float ra = 1.0f - p.s_alpha_s, r4 = 1.0f - p.s_g4, r5 = 1.0f - p.s_g5;
            float cn[7];
            cn[0] = 0.0f;
            cn[1] = ra * (gS[1] - gS[2]) * i1;
            cn[2] = ra * (gS[3] - gS[4]) * i1;
            cn[3] = ra * (gS[5] - gS[6]) * i1;
            cn[4] = r4 * (6.0f * gS[0] - (gS[1] + gS[2] + gS[3] + gS[4] + gS[5] + gS[6]) - 0.75f * Th) * i4;
            cn[5] = r5 * (2.0f * (gS[1] + gS[2]) - (gS[3] + gS[4] + gS[5] + gS[6])) * i5;
            cn[6] = r5 * ((gS[3] + gS[4]) - (gS[5] + gS[6])) * i6;
            add_back7<0>(sg, cn);
        } else {
#pragma unroll
            for (int i = 0; i < 7; ++i) sg[i] = w7(i) * p.dTms;
        }
#pragma unroll
        for (int i = 0; i < 7; ++i) spost[(long long)i * p.ncols + col] = sg[i];
    }
    if (jn >= H) {  // fully liquid column: no ghost node
        if (SPEC && move && jn != jsc) flip_column<ST, FACE>(p, F, js, infl, col, jsc, jn);
        return jn;
    }
    const int kg = guarded_node(fn);
    const float dy = ghost_distance(fn, jn);
    float Tg;
    if (kg < 0) {
        Tg = Tm + (Tm - Tw) * (dy / (float)sn);
    } else {
        float Tk;
        if (kg == k) Tk = y1;
        else if (kg == k - 1 && k >= 1) Tk = y0;
        else if (spec && kg == L) Tk = sum_T(p, gL);
        else Tk = node_T<ST, FACE>(p, G, col, kg, infl, thw);
        Tg = Tm + (Tm - Tk) * (dy / guarded_distance(fn));
    }
    // ghost populations (FP32, like the collision): rest equilibrium at the
    // ghost temperature plus the non-equilibrium part N^-1 (I - Q)(n - n^eq)
    // of the post-collision populations of the liquid node below
    float gh[7];
    const float dTg = Tg - p.Ts;
#pragma unroll
    for (int i = 0; i < 7; ++i) gh[i] = w7(i) * dTg;
    if (jn >= 1) {
        if (!(spec && jn == jsc)) {  // the count changed: the source node moved
            int x, y, z;
            column_node<FACE>(p, col, jn - 1, x, y, z);
            gather_g<ST, FACE>(p, G, x, y, z, infl, thw, gL);
            const bool newly_liquid = (jn - 1) >= jsc;
            if (newly_liquid) {
#pragma unroll
                for (int i = 0; i < 19; ++i) fL[i] = 0.0f;
            } else {
                gather_f<ST, FACE, SPEC>(p, F, js, x, y, z, infl, fL);
            }
        }
        float Th = 0.0f, jx = 0.0f, jy = 0.0f, jz = 0.0f;
#pragma unroll
        for (int i = 0; i < 7; ++i) Th += gL[i];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            jx += ex(i) * fL[i];
            jy += ey(i) * fL[i];
            jz += ez(i) * fL[i];
        }
        const float TL = Th + p.Ts;
        const float ux = jx, uy = jy, uz = jz + 0.5f * p.gbeta * (Th - p.dTms);
        constexpr float i1 = 1.0f / (float)nnorm(1), i4 = 1.0f / (float)nnorm(4);
        constexpr float i5 = 1.0f / (float)nnorm(5), i6 = 1.0f / (float)nnorm(6);
        const float ra = 1.0f - p.s_alpha, r4 = 1.0f - p.s_g4, r5 = 1.0f - p.s_g5;
        float cn[7];
        cn[0] = 0.0f;
        cn[1] = ra * ((gL[1] - gL[2]) - ux * TL) * i1;
        cn[2] = ra * ((gL[3] - gL[4]) - uy * TL) * i1;
        cn[3] = ra * ((gL[5] - gL[6]) - uz * TL) * i1;
        cn[4] = r4 * (6.0f * gL[0] - (gL[1] + gL[2] + gL[3] + gL[4] + gL[5] + gL[6]) - 0.75f * Th) * i4;
        cn[5] = r5 * (2.0f * (gL[1] + gL[2]) - (gL[3] + gL[4] + gL[5] + gL[6])) * i5;
        cn[6] = r5 * ((gL[3] + gL[4]) - (gL[5] + gL[6])) * i6;
        add_back7<0>(gh, cn);
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) gpost[(long long)i * p.ncols + col] = gh[i];
    if (SPEC && move && jn != jsc) flip_column<ST, FACE>(p, F, js, infl, col, jsc, jn);
    return jn;
}

// 4 blocks of 128 a multiprocessor (128 registers: 608 blocks cover a 256 x
// 256 front at once; without the cap, 136 and 192 registers, the loop of
// single 256^3 steps lost 2.5 us a step to a second wave).
//
// jmax (may be null): running maximum of the liquid counts.  A warp whose
// columns exceed it (few do: a count grows by one now and then) raises it with
// an atomic, and its copy in page-locked host memory, jmax_host, which the
// host reads now and then to bound the height of the stream-collide
// grid (nodes two above every neighbouring count are deep solid and do
// nothing).
template <typename ST, int FACE>
__global__ void __launch_bounds__(128, 4) k_front(const __grid_constant__ KP p, ST *__restrict__ F, const ST *G,
                                               const int *__restrict__ js, int *__restrict__ js_next,
                                               int *__restrict__ nb_next,
                                               const double *__restrict__ s, double *__restrict__ s_next,
                                               float *__restrict__ gpost, const float *__restrict__ thw,
                                               int inflight, int move, int *__restrict__ status,
                                               int *jmax, int *jmax_host) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    int jn = -1;
    const int top = jmax ? ld_l2(jmax) : 1 << 30;  // of the steps before
    if (col >= p.ncols) step_launch_wait();
    else jn = front_column<ST, FACE>(p, F, G, js, js_next, nb_next, s, s_next, gpost, thw, inflight, move, status, col);
    // blocks are whole warps and every thread of the grid reaches this point
    const int m = __reduce_max_sync(0xffffffffu, jn);
    if ((threadIdx.x & 31) == 0 && m > top) {
        atomicMax(jmax, m);
        atomicMax_system(jmax_host, m);
    }
}

// The front update with heat conduction in the solid.  4 blocks of 128 an SM
// like k_front: uncapped (168 to 192 registers) a 256 x 256 front took two
// waves, 23.3 against 16.2 us under the profiler, 353 against 348 us a step.
template <typename ST, int FACE>
__global__ void __launch_bounds__(128, 4) k_front_cond(const __grid_constant__ KP p, ST *__restrict__ F,
                                                    const ST *G, const int *__restrict__ js,
                                                    int *__restrict__ js_next, int *__restrict__ nb_next,
                                                    const double *__restrict__ s,
                                                    double *__restrict__ s_next, float *__restrict__ gpost,
                                                    float *__restrict__ spost, const float *__restrict__ thw,
                                                    int inflight, int move, int *__restrict__ status) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= p.ncols) step_launch_wait();
    else
        front_column<ST, FACE, true, true>(p, F, G, js, js_next, nb_next, s, s_next, gpost, thw, inflight, move, status, col,
                                           spost);
}


// ----------------------------------------------------- outputs and inputs
// T and u per node (solid: Tm, or its own temperature with heat conduction
// in the solid, and u = 0), natural values.
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_macro(const __grid_constant__ KP p, const ST *__restrict__ F, const ST *__restrict__ G,
                                               const int *__restrict__ js, const int *__restrict__ js_old,
                                               const float *__restrict__ thw,
                                               int inflight, float *__restrict__ T, float *__restrict__ u) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long c = node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z), col = column<FACE>(p, x, y, z);
    float Tc = p.Tm, ux = 0.0f, uy = 0.0f, uz = 0.0f;
    if (a < js[col]) {
        float g[7], f[19];
        gather_g<ST, FACE>(p, G, x, y, z, inflight != 0, thw, g);
        float Th = 0.0f;
        if (u) gather_f_now<ST, FACE>(p, F, js, js_old, x, y, z, inflight != 0, f);
#pragma unroll
        for (int i = 0; i < 7; ++i) Th += g[i];
        if (u) {
#pragma unroll
            for (int i = 0; i < 19; ++i) { ux += ex(i) * f[i]; uy += ey(i) * f[i]; uz += ez(i) * f[i]; }
            uz += 0.5f * p.gbeta * (Th - p.dTms);
        }
        Tc = p.Ts + Th;
    } else if (p.cond) {
        float g[7];
        gather_g<ST, FACE>(p, G, x, y, z, inflight != 0, thw, g);
        Tc = sum_T(p, g);
    }
    if (T) T[c] = Tc;
    if (u) { u[3 * c] = ux; u[3 * c + 1] = uy; u[3 * c + 2] = uz; }
}

// Natural (unshifted) distributions out, direction-major with stride N.
// Solid nodes report f = 0; deep solid nodes (see deep_solid) report g at
// rest at Tm, the value their slots would hold if they were updated.
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_state_out(const __grid_constant__ KP p, const ST *__restrict__ F, const ST *__restrict__ G,
                                                   const int *__restrict__ js, const int *__restrict__ js_old,
                                                   const int *__restrict__ nb,
                                                   const float *__restrict__ thw, int inflight,
                                                   float *__restrict__ fo, float *__restrict__ go) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long c = node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z), col = column<FACE>(p, x, y, z);
    if (go) {
        float g[7];
        if (a >= js[col] && deep_solid(p, a, nb[col])) {
#pragma unroll
            for (int i = 0; i < 7; ++i) g[i] = w7(i) * p.dTms;
        } else {
            gather_g<ST, FACE>(p, G, x, y, z, inflight != 0, thw, g);
        }
#pragma unroll
        for (int i = 0; i < 7; ++i) go[i * p.N + c] = g[i] + w7(i) * p.Ts;
    }
    if (fo) {
        float f[19];
        const bool liq = a < js[col];
        if (liq) gather_f_now<ST, FACE>(p, F, js, js_old, x, y, z, inflight != 0, f);
#pragma unroll
        for (int i = 0; i < 19; ++i) fo[i * p.N + c] = liq ? f[i] + w19(i) : 0.0f;
    }
}

// New fronts (s_in: an array of ncols heights) and their liquid counts; the
// running maximum of the counts and its copy start anew.
static __global__ void __launch_bounds__(128) k_set_fronts(const double *s_in, int ncols, int H, double *s, int *js,
                                                           int *jmax, int *jmax_host) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col == 0) *jmax = *jmax_host = 0;
    if (col >= ncols) return;
    const double v = s_in[col];
    s[col] = v;
    js[col] = liquid_count(front_pos(v, H), H);
}

// Natural distributions in; leaves the natural layout.  A solid node's own
// populations never enter the method (its post-collision values are reset
// every step): its g is stored at rest at Tm (with heat conduction in the
// solid it keeps its g), and its f slots, which nothing reads before they are
// written, are left alone (they were two thirds of the bytes of an upload
// with a thin layer: 101 -> 48 us at 128^3, front at 0.1 H, with the rest of
// this call).
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_state_in(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                                  const int *__restrict__ js, const float *__restrict__ fi,
                                                  const float *__restrict__ gi) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long c = node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z), col = column<FACE>(p, x, y, z);
    const bool liq = a < js[col];
    if (gi)
#pragma unroll
        for (int i = 0; i < 7; ++i)
            Store<ST>::st(G + i * p.ld + c, (liq || p.cond) ? gi[i * p.N + c] - w7(i) * p.Ts : w7(i) * p.dTms);
    if (fi && liq)
#pragma unroll
        for (int i = 0; i < 19; ++i) Store<ST>::st(F + i * p.ld + c, fi[i * p.N + c] - w19(i));
}

// Initial state: fh = 0 everywhere (rest, rho = 1); g at rest at the given
// profile T(a) below the front and at Tm above (at the profile everywhere
// with heat conduction in the solid).
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_init(const __grid_constant__ KP p, ST *__restrict__ F, ST *__restrict__ G,
                                              const int *__restrict__ js, const float *__restrict__ Tprof) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long c = node_index(p, x, y, z);
    const int a = axial<FACE>(x, y, z), col = column<FACE>(p, x, y, z);
    const float dT = (a < js[col] || p.cond) ? Tprof[a] - p.Ts : p.dTms;
#pragma unroll
    for (int i = 0; i < 19; ++i) Store<ST>::st(F + i * p.ld + c, 0.0f);
#pragma unroll
    for (int i = 0; i < 7; ++i) Store<ST>::st(G + i * p.ld + c, w7(i) * dT);
}

// ---------------------------------------------------------- Nusselt number
// Heat-surface Nusselt number per column (section 3.2, Fig. 4(b)):
// Nu = -H (dT/da at the heated wall) / (Th - Tm), from the heat the last
// streaming carried through the wall link of the column's first node,
// q = in - out = -alpha dT/da, times scale = H / (alpha (Th - Tm)).  The
// link is anti-bounce-back, in = -out + 2 w (Tw - Tm) in shifted values, so
// slot +a of the node gives q alone: in the natural layout it holds `in`
// (q = 2 (in - w (Tw - Tm))); in flight it still holds `out`, the node's
// post-collision population towards the wall (q = 2 (w (Tw - Tm) - out)).
// Tw is the wall field of that streaming.  FP64 from the stored value.
template <typename ST, int FACE>
__device__ __forceinline__ double column_nusselt(const KP &p, const ST *G, const float *thw, int inflight, double scale,
                                                 int col) {
    int x, y, z;
    column_node<FACE>(p, col, 0, x, y, z);
    constexpr int up = FACE == 0 ? 3 : 5;  // the D3Q7 direction leaving the heated wall
    const double v = (double)Store<ST>::ld(G + up * p.ld + node_index(p, x, y, z));
    const double wt = (double)w7(up) * ((double)thw[col] - (double)p.Ts);
    return (inflight ? 2.0 * (wt - v) : 2.0 * (v - wt)) * scale;
}
template <typename ST, int FACE>
__global__ void __launch_bounds__(128) k_nusselt(const __grid_constant__ KP p, const ST *__restrict__ G,
                                                 const float *__restrict__ thw, int inflight, double scale,
                                                 double *__restrict__ nu) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col < p.ncols) nu[col] = column_nusselt<ST, FACE>(p, G, thw, inflight, scale, col);
}

// ------------------------------------------------------ FP64 reductions
// A sum of FP32 values held as three floats: the error of every addition
// (Knuth's two-sum, exact) goes on to the next, so the sum carries some 72
// bits, more than FP64.  FP64 issues at a small fraction of the FP32 rate
// here: with two FP64 sums a node a totals call on a convecting 256^3 state at 0.4 H
// took 165.6 us, with these 150.3 (in flight 198; two floats, which hold only
// 48 bits, 150.4 and 193).
struct TripleSum {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    static __device__ __forceinline__ float two_sum(float &s, float v) {
        const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z));
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(float v) { c = __fadd_rn(c, two_sum(b, two_sum(a, v))); }
    __device__ __forceinline__ double value() const {
        const double tail = (double)b + (double)c;
        return isfinite(tail) ? (double)a + tail : (double)a;  // an infinite a leaves NaN behind
    }
};

constexpr int kTotals = 6;       // partials of a block
constexpr int kTotalsRun = 8;    // heights of a tile
// Block partials of the liquid-node totals: sum (T - Tm), sum (rho - 1),
// count, max |u|^2, and of the column sums: fronts, Nusselt numbers.  Blocks
// walk over tiles of 256 columns by kTotalsRun heights in a fixed order:
// deterministic.  max |u|^2 is taken in FP64, as is, of the nodes whose FP32
// value comes within its rounding (below 4e-7 relative) of the maximum so
// far.  Read bandwidth bounds it (104 bytes a liquid node with FP32 storage);
// with every |u|^2 and count in FP64 too, 64-bit divisions for the node's
// coordinates and the column sums left to one block, a totals call on a 256^3
// cavity at 0.4 H took 486 us (FP16 storage 1127), now 150 (138), in flight 198.
template <typename ST, int FACE>
__global__ void __launch_bounds__(256, 4) k_totals_part(const __grid_constant__ KP p, const ST *__restrict__ F, const ST *__restrict__ G,
                                                     const int *__restrict__ js, const int *__restrict__ js_old,
                                                     const double *__restrict__ s, const float *__restrict__ thw,
                                                     const float *__restrict__ thw_nu, int inflight, double nu_scale,
                                                     double *__restrict__ part) {
    __shared__ double sh[kTotals][256];
    TripleSum sT, sr;
    double ss = 0.0, sn = 0.0, umax = 0.0;
    float ufloor = 0.0f;  // nodes with an FP32 |u|^2 below it are not the maximum
    int n = 0;
    const int ctiles = (p.ncols + 255) / 256, atiles = (p.H + kTotalsRun - 1) / kTotalsRun;
    const long long tiles = (long long)ctiles * atiles;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int at = (int)(t / ctiles), col = (int)(t - (long long)at * ctiles) * 256 + (int)threadIdx.x;
        if (col >= p.ncols) continue;
        if (at == 0) {
            ss += s[col];
            sn += column_nusselt<ST, FACE>(p, G, thw_nu, inflight, nu_scale, col);
        }
        const int a0 = at * kTotalsRun, jc = js[col], a1 = a0 + kTotalsRun < jc ? a0 + kTotalsRun : jc;
#pragma unroll 1
        for (int a = a0; a < a1; ++a) {
            int x, y, z;
            column_node<FACE>(p, col, a, x, y, z);
            float g[7], f[19];
            gather_g<ST, FACE>(p, G, x, y, z, inflight != 0, thw, g);
            gather_f_now<ST, FACE>(p, F, js, js_old, x, y, z, inflight != 0, f);
            float Th = 0.0f, rh = 0.0f, ux = 0.0f, uy = 0.0f, uz = 0.0f;
#pragma unroll
            for (int i = 0; i < 7; ++i) Th += g[i];
#pragma unroll
            for (int i = 0; i < 19; ++i) { rh += f[i]; ux += ex(i) * f[i]; uy += ey(i) * f[i]; uz += ez(i) * f[i]; }
            uz += 0.5f * p.gbeta * (Th - p.dTms);
            sT.add(Th - p.dTms);
            sr.add(rh);
            ++n;
            if (ux * ux + uy * uy + uz * uz >= ufloor) {
                const double u2 = (double)ux * ux + (double)uy * uy + (double)uz * uz;
                if (u2 > umax) {
                    umax = u2;
                    ufloor = (float)(u2 * (1.0 - 1e-6));
                }
            }
        }
    }
    const double v[kTotals] = {sT.value(), sr.value(), (double)n, umax, ss, sn};
#pragma unroll
    for (int k = 0; k < kTotals; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
#pragma unroll
            for (int k = 0; k < kTotals; ++k)
                sh[k][threadIdx.x] = k == 3 ? fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + w])
                                            : sh[k][threadIdx.x] + sh[k][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x < kTotals) part[blockIdx.x * kTotals + threadIdx.x] = sh[threadIdx.x][0];
}

// Final pass in one block: out = {liquid fraction, sum (T - Tm), sum (rho - 1),
// liquid nodes, max |u|, sum s, mean Nusselt number over the heated wall};
// with t >= 0 also writes the time first.
static __global__ void __launch_bounds__(256) k_totals_final(const double *__restrict__ part, int nparts, int ncols,
                                                      double H, double t, double *__restrict__ out) {
    __shared__ double sh[kTotals][256];
    double v[kTotals] = {};
    for (int b = threadIdx.x; b < nparts; b += blockDim.x) {
#pragma unroll
        for (int k = 0; k < kTotals; ++k)
            v[k] = k == 3 ? fmax(v[k], part[b * kTotals + k]) : v[k] + part[b * kTotals + k];
    }
#pragma unroll
    for (int k = 0; k < kTotals; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
#pragma unroll
            for (int k = 0; k < kTotals; ++k)
                sh[k][threadIdx.x] = k == 3 ? fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + w])
                                            : sh[k][threadIdx.x] + sh[k][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double *o = out;
        if (t >= 0.0) *o++ = t;
        o[0] = sh[4][0] / (H * (double)ncols);
        o[1] = sh[0][0];
        o[2] = sh[1][0];
        o[3] = sh[2][0];
        o[4] = sqrt(sh[3][0]);
        o[5] = sh[4][0];
        o[6] = sh[5][0] / (double)ncols;
    }
}

}  // namespace lbm

// handle.h -- internal definition of the cavity handle (opaque in the C ABI),
// shared by the single-cavity entry points and the ensemble.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "../../include/lbm_melt.h"
#include "lbm_core.cuh"

// Lattice parameters derived from the problem statement (section 1, Eq. 7).
struct Derived {
    int H, P1, P2;
    long long N, ncols;
    double nu, alpha, gbeta, s_nu, s_alpha, lambda, t0, s0;
    double s_e, s_eps, s_q, s_pi, s_m, s_g4, s_g5;
};

struct lbm_melt {
    lbm::KP kp;
    lbm::Links lk;     // interior link offsets of the odd step
    Derived d;
    int face, precision;
    double Ste, Th, Tc, Tm;
    cudaStream_t stream;
    int device;
    void *F, *G;
    int *js[2];
    int *nb[2];
    double *s[2];
    int cur;
    float *gpost;
    float *thw_cur, *thw_prev;
    int thw_pending;   // set_hot_wall happened while values were in flight
    long long thw_gen; // number of set_hot_wall calls (a recorded run keeps the field of its record)
    int thw_last_prev; // set_hot_wall since the last step in the natural layout: thw_prev holds the
                       // field of the last streaming (the Nusselt number's wall value)
    double *nu_dev;    // per-column Nusselt numbers (ncols)
    double *sum_dev;
    unsigned int *ticket;  // last-block ticket of the one-launch column sum (k_sum_once)
    double *red_part;  // scratch: per-block partials of the FP64 totals
    int nred;          // number of partial blocks
    double *totals_dev;  // 7 doubles
    double *report;    // ring of report rows (8 doubles: t, totals)
    long long report_every, report_cap, report_rows;
    int inflight;      // last stream-collide was an even (local) step
    long long steps;
    size_t bytes;
    int timing;
    int bx, by;        // block shape of the per-node kernels (0: default)
    int cblk;          // threads per block of the per-column kernels
    int sms;           // SMs of the device
    // The stream's last work wrote what the step's kernels load early: the next
    // one is launched plainly (take_plain).  plain_capture: the capture whose
    // first step already was.
    int plain_next;
    unsigned long long plain_capture;
    // Running maximum of the liquid counts, kept by k_front on the device;
    // stream-collide blocks at heights >= it + 3 (all deep solid) return at
    // once.  The front kernels (the ensemble's too) raise a copy in page-locked
    // memory with it, and the host records an event every kRbEvery steps;
    // before a stream-collide the host takes the newest event at least kRbLag
    // steps old (waiting for it only when it runs that far ahead of the
    // device) and launches no block above the maximum it then reads + the
    // event's age + 2 (a count grows by at most one node per step).
    static const int kRbRing = 32, kRbLag = 16, kRbEvery = 4;
    int *jmax_dev;
    // Page-locked, written by the kernels and read by the host once the stream
    // has got there: the front status (kStatus, touched on an error only), the
    // running maximum (kTop), then small results of the synchronising calls.
    // With device flags copied back by each such call (an ensemble: by each
    // member), 16 steps of 8 FP16 cavities with restores and reads took 840 us
    // instead of 737, a 256^3 readout 396 instead of 374.
    static const int kStatus = 0, kTop = 1, kHostOut = 8;
    int *flags;
    double *host_out;
    cudaEvent_t rb_ev[kRbRing];
    long long rb_step[kRbRing];  // exec step after which each event was recorded
    long long rb_next;           // events recorded so far
    long long rb_valid_from;     // events before this one are not bounds any more
    long long rb_synced;         // newest event known complete
    long long exec_steps;        // steps this handle executed (never rewound)
    double Ra;         // as given to create
    int derived_from_Ra;
    // Heat conduction in the solid (lbm_melt_set_solid_conduction): the
    // conductivity ratio k_s / k_l (0: off, the solid held at Tm) and the
    // solid side's ghost populations of each column (7 x ncols).
    double ks_kl;
    float *spost;
    int member;        // owned by an ensemble (whose kernel holds the solid at Tm)
    void *tape;        // recorded run for the adjoint (adjoint.cu)
    void *adj_ws;      // the adjoint's device buffers, kept between gradients (adjoint.cu)
    // Steps replayed from CUDA graphs (lbm_melt_step): graph_steps steps per
    // replay (0: every step launched on its own).  One instantiated graph per
    // starting (cur, inflight) phase; each records the stream-collide grid
    // height and block shape it was captured with.
    int graph_steps;
    // Nodes per thread of the stream-collide: -1 chooses (two for cavities
    // above 160^3 with an even nx, one otherwise), 0 one, 1 two (even nx).
    int pairs_mode;
    cudaStream_t cap_stream;     // private stream the graphs are captured on
    struct StepGraph {
        cudaGraphExec_t exec;
        int height, bx, by, linear;
    } graphs[2][2];              // [cur][inflight]
    std::vector<cudaEvent_t> ev;  // start/stop pairs of timed launches
    size_t ev_used;
    char err[512];
};

// Release a handle's recorded run and the adjoint's buffers (defined with
// the adjoint).
void lbm_tape_free(lbm_melt *h);
// Enqueue one step (stream-collide, front with flip) from phase (cur, inflight)
// on stream st, the stream-collide grid cut at `height`; advances cur and
// inflight.  No host bookkeeping (step counters, read-backs, report rows).
// snap (may be null, else lbm_step_snapshots holds): the stream-collide also
// writes the snapshot of the state it starts from.
namespace lbm { struct SnapOut; }
cudaError_t lbm_enqueue_step(lbm_melt *h, int &cur, int &inflight, int height, cudaStream_t st,
                             const lbm::SnapOut *snap = nullptr);
bool lbm_step_snapshots(lbm_melt *h);
// Reads the sticky front status on the handle's stream (synchronises):
// LBM_EUNSTABLE after a step with |ds| > 1/2, LBM_ENAN after a non-finite
// front temperature, else LBM_OK.
lbm_status lbm_check_status(lbm_melt *h);


// Internal layout shared by the host side (opf_api.cu) and the kernels
// (opf_kernels.cu).  Not part of the public ABI.
//
// Numbering: nodes are renumbered by reverse Cuthill-McKee and lines sorted by
// their lower-numbered end (the line's "owner"), so that the two ends of a
// line are processed close together in time; the C ABI converts to and from
// the caller's numbering on import and export.  Devices keep the caller's
// order (generators, loads, batteries).
//
// Device memory layout (structure of arrays, time innermost so that every row
// of T floats is one contiguous, 16-byte aligned segment when T % 4 == 0):
//   lines   P, MID, V1, V2                  2 x [L][Kp][T] float (double buffer)
//   nodes   U, PU = pbar + u, THBAR         2 x [N][Kp][T] float (double buffer)
// (line- and node-major: the K+1 contingency rows of one line or node are
// one contiguous run, so the node sums gather long runs per terminal)
//   devices PD, DPD                         [S][T]         float
//   inner ADMM state of ramp generators     lam, beta [n_ramp][4][T],  q [n_ramp][3][T]
//   inner ADMM state of batteries           lam, beta [n_stor][9][T+1], q [n_stor][3][T+1]
// (q: pivots; 1 / q and -off / q beside them where the shared-memory form
// solved last or since they were factored, else 0 for the first 1 / q)
// Buffer (it & 1) holds the state after `it` iterations; an iteration reads
// the old buffers and writes the other ones, because both ends of a line
// evaluate its prox from the old line and node values.
// V1/V2 hold the phase duals one step behind: the update v += theta - theta_bar
// of iteration i is folded into the line pass of iteration i+1, which already
// reads theta and theta_bar (so v is read and written once per iteration).
#ifndef OPF_INTERNAL_H_
#define OPF_INTERNAL_H_

#include <stddef.h>
#include <stdint.h>

namespace opfk {

// threads per CTA of the iteration kernels
constexpr int BLOCK = 256;

// residual partial-sum slots.  SL_NF counts non-finite node values: the prox
// clamps (fminf/fmaxf) would otherwise turn a NaN input into a finite bound.
enum { SL_PP = 0, SL_PT = 1, SL_DP = 2, SL_DT = 3, SL_NF = 4, NSLOT = 5 };

// The scalars of the current iteration in the form the iteration kernels read
// them: two 16-byte loads per thread, with no barrier, conversion or 64-bit
// remainder in front of a kernel's first load of the state.  Every writer of
// DevScalars keeps it in step (set_iter).
struct alignas(16) Iter {
  float frp, frt, fsu, fsv;   // penalties, pending rescales of u and v
  float rho_dev;              // rho' = (K+1) rho_p
  int old;                    // buffer of the previous iterate (it & 1)
  int flags;                  // ITF_*
  int left;                   // iterations before the next one that forms residuals (0: this one)
};
enum {
  ITF_SKIP = 1,      // stopped in this call (passed stopping test, stall) or a sticky error: return at once
  ITF_RES = 2,       // the residuals are read (stopping test, adaptation, end of the call)
  ITF_VFRESH = 4     // V1/V2 already hold the current v
};

// Scalars that persist on the device between launches.
struct DevScalars {
  double rho_p, rho_th;  // penalties in force for the next iteration
  double su, sv;         // pending rescale of u and v (1 = none), applied on next read
  double res[6];         // residuals of the last iteration
  long long it;          // iterations run
  int converged;
  int status;            // sticky opf_status from the device (0 = ok)
  int v_fresh;           // 1: V1/V2 already hold the current v (after import / reset)
  int stop;              // set by the decision kernel (passed stopping test, error);
                         // cleared at the start of every opf_iterate call
  long long it_last;     // the last iteration of the current call: residuals are formed
                         // there and at stopping-test and adaptation iterations only
  // stall rule (opf_options.stall_window): best max(||r_primal||, ||r_dual||)
  // at a stopping test and its iteration; the iteration at which the rule
  // fixed the penalties (0 = they still adapt); 1 after a stall at fixed
  // penalties (stops the call; the next opf_iterate restarts the window)
  double stall_ref;
  long long stall_it;
  long long frozen_at;
  int stalled;
  int pad0;
  long long hist_n;      // residual-history rows written (ring of Params::hist_cap rows)
  Iter cur;              // the next iteration's scalars (set_iter)
};

// Battery group offsets inside lam/beta rows of stride Tp = T + 1.
enum { SG_E1 = 0, SG_E2 = 1, SG_E3 = 2, SG_CU = 3, SG_CL = 4, SG_DU = 5, SG_DL = 6,
       SG_SU = 7, SG_SL = 8, SG_N = 9 };
// Ramp-generator groups, stride T.
enum { RG_UP = 0, RG_LO = 1, RG_RU = 2, RG_RD = 3, RG_N = 4 };

struct Params {
  int N, L, T, Kp, S;
  int n_dnode, n_ramp, n_stor;
  int n_hvdc, hvdc0;                     // HVDC links; device id of the first link's terminal 1
  // lines (internal numbering)
  const int *line_n1, *line_n2;  // internal node of terminal 1 (from) and terminal 2 (to)
  const float *line_b, *line_u;
  const int *out_line;  // [Kp], internal index of the outaged line, -1 = none
  // double-buffered line state: terminal-2 power p, the mean terminal angle
  // mid (theta_{1,2} = mid +- p / (2b), the line prox keeps theta1 - theta2 =
  // p / b; the outaged line of a contingency has p = 0 and stores its half
  // angle difference in p's place), and the phase duals
  float *P[2], *MID[2], *V1[2], *V2[2];
  // nodes (internal numbering), double-buffered
  float *U[2], *PU[2], *THBAR[2];   // PU = pbar + u (unscaled): what the proxes read
  // incident lines of each node: x = 2*l + end (end 1: the node is terminal 2), y = other node
  const int *lcsr_ptr;
  const int2 *lcsr;
  const int *dcsr_ptr, *dcsr_idx;  // devices of each node
  const float *cnt_p, *cnt_th;     // terminals per node: all (power), line terminals (phase)
  const float *rcnt_p, *rcnt_th;   // their reciprocals (0 for a node without line terminals)
  // per node, 3 int4: (cnt_p, cnt_th, rcnt_p, rcnt_th as float bits), the first
  // four line-terminal codes 2*l + end (-1 = none), (tcode begin, end of the
  // rest, device count, first of the node's entries in dcsr_idx)
  const int4 *nrec;
  const int4 *ndev4;               // each node's first four devices
  const int *tcode;                // line-terminal codes beyond the first four per node,
                                   // each node's list padded to a multiple of 4 with -1
  // per node and time step, over the node's devices (the same in every
  // contingency): sum of p_d, and the Welford mean and sum of squared
  // deviations of the change of p_d in this iteration
  float *DSP, *DSM, *DSQ;          // [N][T]
  // devices: type 0 = closed-form prox clip((rho X - b)/(2a + rho), lo, hi), 1 = inner ADMM
  float *PD, *DPD;
  const int *dev_node, *dev_type;
  // nodes with devices; per node its closed-form devices and whether it has
  // inner-ADMM devices, whose input avg_k(pbar + u) is then kept in XS
  const int *dnode_ids, *dnode_ptr, *dnode_dev, *dnode_keep;
  // nodes with closed-form devices: (node, first and one past the last entry of dnode_dev, 0)
  const int4 *crec;
  int n_cnode;
  float *XS;  // [N][T], avg_k(pbar + u) of the previous iterate at kept nodes
  const float *dev_a, *dev_b;
  const float *dev_lo, *dev_hi;  // [S][T]
  // inner-ADMM devices in the order of their warps (batteries, ramp-limited
  // generators): (device, node) and a battery's (efficiency, power, duration,
  // cost) or a generator's (a, b, ramp limit, 0)
  const int2 *irec;
  const float4 *ipar;
  // ramp-limited generators
  const int *ramp_ids;
  const float *ramp_R;
  float *ramp_lam, *ramp_beta, *ramp_q, *ramp_rho;
  // batteries
  const int *stor_ids;
  const float *stor_eff, *stor_P, *stor_dur, *stor_cost;
  const float *hvdc_u;                   // [n_hvdc]; link h has terminals hvdc0 + 2h, hvdc0 + 2h + 1
  float alpha;                           // over-relaxation (Section 3.6); 1 = plain message passing
  float *stor_lam, *stor_beta, *stor_q, *stor_rho, *stor_delta;  // delta [n_stor][T]
  // numbering maps (internal -> caller) for import / export
  const int *node_perm, *line_perm;
  // scratch
  double *partials;  // [node_grid][NSLOT] residual partial sums of the node kernel (one per CTA of its own grid)
  int node_grid;     // CTAs of the node kernel (partial-sum slots)
  float *wsums;      // [node_grid][BLOCK / 32][NSLOT] in a batch: their parts by warp
  unsigned *done;    // CTAs of the node kernel that have finished this iteration (0 between iterations)
  DevScalars *sc;
  // options
  double eps, mu, gamma, tol;
  int adapt_every, check_every, inner_iters;
  int stall_window;     // 0 = no stall rule
  long long adapt_until;  // last iteration that may adapt (0 = no limit)
  double *hist;         // residual history ring [hist_cap][HIST_COLS]
  int hist_cap;
  // contingency slice (opf_create_slice): this context holds contingencies
  // k_base .. k_base + Kp - 1 of Kp_glob; the sums over k that couple them
  // (Section 3.2 step 2) and the residual sums (Section 3.3) go through the
  // exchange buffer xsum, which the caller sums over the slices:
  //   [n_dnode][T] sum_k (pbar + u) at the nodes with devices,
  //   [n_dnode][T] sum_k u there (on adaptation iterations; else 0),
  //   [NSLOT] residual partial sums
  int Kp_glob;          // K + 1 of the whole problem (= Kp without slices)
  int k_base;
  int slice;            // 1: a slice context
  double *xsum;
};

// columns of a residual-history row (include/opf.h, opf_history)
constexpr int HIST_COLS = 10;
enum { HF_CONVERGED = 1, HF_ADAPTED = 2, HF_FROZEN = 4, HF_STALLED = 8, HF_NONFINITE = 16 };

// offsets of element (contingency k, line l / node n, step t)
__host__ __device__ __forceinline__ size_t lidx(const Params &p, int k, int l, int t) {
  return ((size_t)l * p.Kp + k) * p.T + t;
}
__host__ __device__ __forceinline__ size_t nidx(const Params &p, int k, int n, int t) {
  return ((size_t)n * p.Kp + k) * p.T + t;
}

// whether the penalties may still change after iteration itn (1-based):
// adaptation on, within opf_options.adapt_until, not fixed by the stall rule
__host__ __device__ __forceinline__ bool adapting(const Params &p, const DevScalars &sc, long long itn) {
  return p.adapt_every > 0 && (p.adapt_until <= 0 || itn <= p.adapt_until) && sc.frozen_at == 0;
}
// iteration itn adapts the penalties (Section 3.5, every adapt_every iterations)
__host__ __device__ __forceinline__ bool adapt_at(const Params &p, const DevScalars &sc, long long itn) {
  return adapting(p, sc, itn) && itn % p.adapt_every == 0;
}
// iteration itn forms its residuals
__host__ __device__ __forceinline__ bool res_at(const Params &p, const DevScalars &sc, long long itn) {
  return adapt_at(p, sc, itn) || (p.eps > 0 && p.check_every > 0 && itn % p.check_every == 0) || itn >= sc.it_last;
}
// the next iteration's scalars from the persistent ones
__host__ __device__ __forceinline__ void set_iter(const Params &p, DevScalars &sc) {
  Iter r;
  r.frp = (float)sc.rho_p;
  r.frt = (float)sc.rho_th;
  r.fsu = (float)sc.su;
  r.fsv = (float)sc.sv;
  r.rho_dev = (float)(p.Kp_glob * sc.rho_p);
  r.old = (int)(sc.it & 1);
  // the first of the next iterations it + 1 .. it_last that forms residuals:
  // the call's last one, a stopping test, or an adaptation
  long long left = sc.it_last - (sc.it + 1);
  if (p.eps > 0 && p.check_every > 0) {
    const long long c = p.check_every - 1 - sc.it % p.check_every;
    if (c < left) left = c;
  }
  if (p.adapt_every > 0) {
    const long long a = p.adapt_every - 1 - sc.it % p.adapt_every;
    if (a < left && adapting(p, sc, sc.it + 1 + a)) left = a;
  }
  r.left = (int)(left > 0 ? left : 0);   // a call has at most 2^31 - 1 iterations
  r.flags = ((sc.status != 0 || sc.stop != 0) ? ITF_SKIP : 0) | (r.left == 0 ? ITF_RES : 0) |
            (sc.v_fresh ? ITF_VFRESH : 0);
  sc.cur = r;
}

// Launch configuration of one iteration's kernels.
struct IterPlan {
  int line_grid, node_grid;            // 0: the kernel has no work
  int line_ipt;                        // line items per thread
  int small;                           // 1: whole iterations on one CTA (opfk_small_launch)
  int node_lat;                        // few node items: all loads of an item requested together
  int fused;                           // 1: one device kernel; 0: averages, inner ADMM and device sums apart
  int dev_inner, dev_closed;           // CTAs of the device kernel for inner-ADMM and (fused) closed-form devices
  int xs_grid, dsum_grid;              // not fused: averages with closed-form devices, device sums
  size_t inner_smem;
  int inner_warps; // warps of a CTA that take inner-ADMM devices
  int inner_c;     // register chunk of the inner-ADMM kernel (0: shared-memory path)
};

// The streams of a batch's phases and the events between them: devices and
// node sums on main, line proxes on aux, and on dev the devices that solve in
// shared memory.
struct Lanes {
  void *main, *aux, *dev;
  void *ev_fork, *ev_join, *ev_dev;
};

// A batch of instances: the CTA schedules of the device and line kernels,
// concatenated in one array of (instance, block within the instance, blocks of
// the instance, 0), in the order of BatchKernel.
enum BatchKernel { BK_SMEM, BK_INNER, BK_CLOSED, BK_LINE4, BK_LINE1, BK_COUNT };
// The node kernel's CTAs are dealt out on the device, over the instances that
// run: one wave of them (slots), each instance's share by its items, so that
// the last running instances of a batch have the GPU to themselves.
struct NodeShare {
  int inst;
  unsigned items;   // node items (of four steps or one)
  int grid;         // at most this many CTAs (its residual partial sums: Params::node_grid)
  int pad;
};
struct NodeDeal {
  const NodeShare *share;  // [n]
  int4 *slot;              // [cap] (instance or -1, block within it, its blocks, 0)
  int *dirty;              // 1: slot is to be written anew
  int n, slots, cap;
};
struct BatchPlan {
  int count[BK_COUNT];
  int offset[BK_COUNT];
  NodeDeal deal;           // n, slots and cap; the caller adds the arrays
  size_t inner_smem;       // of the kernel that solves in shared memory (BK_SMEM)
  int inner_c;             // the largest register chunk of the batch's instances
  int relax;   // the instances run over-relaxed (alpha != 1): the node kernels that carry it
};
// How a batch schedule lays out CTAs: instances in `order` (NULL: as given),
// each instance's CTAs of a phase contiguous or dealt round-robin across
// instances, and `div` times fewer CTAs for the devices, each doing
// proportionally more work.
struct BatchLayout {
  const int *order;
  int interleave;
  int div;
};

}  // namespace opfk

// Launch wrappers implemented in opf_kernels.cu (host callable).
extern "C++" {
// Record the message returned by opf_last_error (opf_api.cu) and pass s on.
int opf_record_error(int s, const char *msg);
// Grids of the iteration kernels for this problem on the current device.
int opfk_plan(const opfk::Params &p, opfk::IterPlan *plan);
// Start a call of n iterations: the residuals are formed at its last one;
// clear_stop restarts a context that stopped (opf_iterate, not batches).
int opfk_begin_launch(const opfk::Params &p, long long n, int clear_stop, void *stream);
int opfk_begin_batch_launch(const opfk::Params *d_params, const opfk::BatchPlan &bp, int n_inst, long long n,
                            void *stream);
// Enqueue one iteration: the device kernel (or xs, inner and dsum) and the
// node kernel (whose last CTA takes the decisions) on main_stream, the line kernel on aux_stream (forked
// after the previous iteration, joined before the node kernel).  Works under
// stream capture.
int opfk_iteration_enqueue(const opfk::Params &p, const opfk::IterPlan &plan, void *main_stream,
                           void *aux_stream, void *ev_fork, void *ev_join);
// n iterations of a small instance (IterPlan::small) in one launch.
int opfk_small_launch(const opfk::Params &p, int n, void *stream);
// Schedules of the batch kernels for n instances (host parameter copies and
// their plans): fills sched (4 ints per CTA, BatchPlan order), share [n] (NULL:
// not wanted) and the plan.
int opfk_batch_plan(const opfk::Params *hp, const opfk::IterPlan *plans, int n, const opfk::BatchLayout &lay,
                    int *sched_out, long long sched_cap, long long *sched_len, opfk::NodeShare *share,
                    opfk::BatchPlan *bp);
// Enqueue one iteration of every instance: d_params [n] and d_sched on the
// device.
int opfk_batch_enqueue(const opfk::Params *d_params, const int *d_sched, const opfk::BatchPlan &bp,
                       const opfk::Lanes &on);
// State import / export between internal and caller numbering; `cur` selects
// the node buffer holding the current state.
int opfk_import_launch(const opfk::Params &p, int cur, const float *p_line, const float *th1,
                       const float *th2, const float *v1, const float *v2, const float *u,
                       void *stream);
// The inner-ADMM state between the device arrays and the caller's layout
// (device pointers, n = opf_info.inner_len); an import wants the arrays
// zeroed and sets the penalty its duals are scaled for (rho, negative).
int opfk_inner_export_launch(const opfk::Params &p, float *out, long long n, void *stream);
int opfk_inner_import_launch(const opfk::Params &p, const float *in, long long n, float rho, void *stream);
int opfk_node_average_launch(const opfk::Params &p, int cur, void *stream);
// Starting state from node rows [T][N][stride] (price / price_scale, angle),
// caller numbering; u = -price * u_scale
int opfk_start_from_nodes_launch(const opfk::Params &p, int cur, const float *rows, int stride,
                                 float price_scale, float u_scale, void *stream);
int opfk_project_v_launch(const opfk::Params &p, int cur, void *stream);
int opfk_export_lines_launch(const opfk::Params &p, int cur, float *p_line, float *th1, float *th2,
                             float *v1, float *v2, void *stream);
// Device powers [S][T] (caller order = internal order) of the actual iterate.
int opfk_export_pdev_launch(const opfk::Params &p, float *out, void *stream);
int opfk_export_nodes_launch(const opfk::Params &p, int cur, float *u, float *theta_node,
                             float *price, void *stream);
// Write the scalars in stream order, from the launch's own copy (nothing to wait for).
int opfk_set_scalars_launch(const opfk::Params &p, const opfk::DevScalars &sc, void *stream);
int opfk_set_rho_launch(const opfk::Params &p, double rho, void *stream);
// Contingency slices: the local half of one iteration (devices from the
// exchanged sums, line proxes, node sums, then this slice's sums into the
// exchange buffer) and the decisions from the exchanged sums; `prime`
// writes the sums of the current state (before the first iteration).
int opfk_slice_local_enqueue(const opfk::Params &p, const opfk::IterPlan &plan, void *main_stream,
                             void *aux_stream, void *ev_fork, void *ev_join);
int opfk_slice_finish_enqueue(const opfk::Params &p, void *stream);
int opfk_slice_prime_launch(const opfk::Params &p, void *stream);
}

#endif  // OPF_INTERNAL_H_

// On-chip evolution for systems whose columns fit in one CTA's shared memory.
//
// One CTA owns a group of Sc state columns for the whole run: the state, the RK4
// stage input and increment (forward) or the co-state, kbar and the stage inputs
// (adjoint) stay in shared memory across steps, so a full forward evolution is one
// launch and an adjoint checkpoint segment is two (recompute, then pull back).
// Columns never exchange data during the evolution (Eq. 1's H(t) acts on each
// column separately), so CTAs need no grid synchronisation; the cross-densities of
// the gradient (Sec. 2.5) are contracted per CTA and stage into per-CTA
// accumulators that one reduction sums in a fixed order.
#pragma once
#include "grad.cuh"
#include "onchip_real.h"

struct OnchipPlan;   // opaque

// nullptr unless the plan is a single tile (one pass of the tiled kernels), every
// mode has the same level count (2..5) and at least one column fits in shared memory
// for the Q2 kernel (onchip_forward_ok / onchip_adjoint_ok tell whether the RK4
// kernels fit too).  K drives and sumd = sum of level counts size the adjoint's
// per-stage buffers.  two_rows: the adjoint pulls back with rows of its own (open systems).
// fwd_only: the columns per CTA are those of the forward kernel (propagators).
// rt (nullable): the terms, when they are real up to the frame phases (interaction frame);
// the forward evolution then runs on the real-operator kernels where they apply.
OnchipPlan* onchip_plan_create(const KPlan& p, bool mixed, int K, int sumd, cudaStream_t st,
                               const OcrTerms* rt = nullptr, bool two_rows = false, bool fwd_only = false);
bool onchip_real(const OnchipPlan* oc);
// The gradient runs on the real-operator kernels too (ocr_densities).
bool onchip_real_adjoint(const OnchipPlan* oc);
const OcrPlan* onchip_real_plan(const OnchipPlan* oc);
void onchip_plan_destroy(OnchipPlan* oc);
// The adjoint kernel fits too (gradient solves may use the on-chip path).
bool onchip_adjoint_ok(const OnchipPlan* oc);
// complex128 entries of one state image (CTA-major, Sc columns of D entries per CTA).
long long onchip_state_elems(const OnchipPlan* oc);
// stage-precision entries of one stored stage-input image (all CTAs).
long long onchip_stage_elems(const OnchipPlan* oc);
int onchip_ctas(const OnchipPlan* oc);
// doubles of one CTA's operator/energy/coupling accumulators (GradAcc layout minus gF).
long long onchip_acc_doubles(const OnchipPlan* oc);

// RK4 steps n0 .. n1-1 in chunks of L steps, all chunks side by side in one launch (L >=
// n1 - n0: one chunk, the serial evolution).  Every chunk starts from its image of img_in
// (chunk-major state images), from the identity (ident: column j in basis state j), or from
// psi_api (D x S, column innermost).  Outputs, where non-null: img_out, the chunks' final
// images; psi_out (API layout, one chunk); ck_out, one chunk, the state before step
// n0 + c K at ck_out + c * state_elems; segY, every stage input of every step (stage images,
// slot 4 (step - n0) + stage).  rev: the steps backwards with their adjoint maps (one
// chunk pulls a co-state from after step n1-1 to before step n0, and ck_out + c *
// state_elems is the co-state after the last step of segment c).  Returns launches.
struct OnchipRealTables {
  const void* coef = nullptr;     // drive coefficients (3N x K) and frame phases (3N x sumd),
  const void* ph = nullptr;       // stage precision
  const double2* opd = nullptr;   // flat truncated operators
  const double* J = nullptr;      // couplings
  const void* half = nullptr;     // onchip_half_step
};
struct OnchipForward {
  const void* tab = nullptr;
  OnchipRealTables rt;            // onchip_real plans
  const double2* psi_api = nullptr;
  const double2* img_in = nullptr;
  double2* img_out = nullptr;
  double2* psi_out = nullptr;
  double2* ck_out = nullptr;
  int K = 1;
  void* segY = nullptr;
  bool ident = false, rev = false;
  bool rows = false;              // the complex-row kernels, also where the plan is real
};
int onchip_forward(const OnchipPlan* oc, const OnchipForward& f, int n0, int n1, int L, double dt, cudaStream_t st);
// f and b over all N steps side by side in one launch (serial passes that do not wait for one
// another: the states, and co-states of a basis).
int onchip_forward_pair(const OnchipPlan* oc, const OnchipForward& f, const OnchipForward& b, int N, double dt,
                        cudaStream_t st);
// nimg images of nin columns -> of the plan's columns in place, out_s = sum_j W[j][s] in_j (W: nin x
// S, device; padding columns become zero); f32: complex64 images, else complex128.
bool onchip_mix_ok(const OnchipPlan* oc, int nin);
cudaError_t onchip_mix(const OnchipPlan* oc, void* img, bool f32, long long nimg, const double2* W, int nin,
                       cudaStream_t st);
// CTAs of the forward (adjoint) launch that one SM holds at once.
int onchip_fwd_resident(const OnchipPlan* oc);
int onchip_adj_resident(const OnchipPlan* oc);
// CTAs of one chunk of the forward launch.
int onchip_fwd_ctas(const OnchipPlan* oc);
// D entries of the stage precision: exp(-i E dt/2) of every composite level.
void onchip_half_step(const OnchipPlan* oc, const double* E, double dt, void* q, cudaStream_t st);
// Columns of a state image, padding included.
int onchip_columns(const OnchipPlan* oc);
void onchip_from_image(const OnchipPlan* oc, const double2* img, double2* api, cudaStream_t st);
// Columns through groups of G consecutive chunk propagators (FP64).  U: C column-major D x D
// matrices, u_stride entries apart.  Group g starts from column image start + g start_stride
// (null: the identity) and, in chunk order (adjoint: reverse order, with U^dag), writes the
// columns before (adjoint: after) chunk c to states + c state_stride and the result to
// last + g last_stride.
struct OnchipChain {
  const double2* U = nullptr;
  const double2* start = nullptr;
  double2* states = nullptr;
  double2* last = nullptr;
  long long u_stride = 0, start_stride = 0, state_stride = 0, last_stride = 0;
  int D = 0, C = 0, G = 1;
  bool adjoint = false;
};
int onchip_chain(const OnchipChain& a, int ncols, int ngroups, cudaStream_t st);
// API layout -> state image (columns past S are zero).
void onchip_to_image(const OnchipPlan* oc, const double2* api, double2* img, cudaStream_t st);
// Per-stage tables the adjoint reads, in the stage precision (complex64 / float in
// mixed precision, complex128 / double otherwise): term rows (3N x row), drive
// coefficients (3N x K), frame phases (3N x sumd) and the flat truncated operators.
struct OnchipTables {
  const void* tab;
  const void* atab;      // rows the co-state is pulled back with (tab unless the plan has two_rows)
  const void* coef;
  const void* ph;
  const void* opd;
};
// Adjoint of steps n0 .. n1-1 in chunks of L steps, side by side in one launch, from the
// stage inputs in segY: chunk c pulls its co-state image lam + c * state_elems (the co-state
// after its last step) back in place; the cross-densities of every stage are contracted into
// gF_cta (CTA-major, 3N x K each, one store per stage slot) and acc_cta (chunk- and
// CTA-major, onchip_acc_doubles each, added to).  *err is set when a bounded wait on a bulk
// copy gives up.  Returns launches.
// colow: when onchip_colow_global(oc), a device buffer of onchip_state_elems complex64
// entries per chunk for the low words of the float-float co-state; else null.
int onchip_adjoint(const OnchipPlan* oc, const OnchipTables& tb, const void* segY, double2* lam, int n0, int n1,
                   int L, double dt, const XArgs& xa, int nst, double* gF_cta, double* acc_cta, int* err,
                   void* colow, cudaStream_t st);
bool onchip_colow_global(const OnchipPlan* oc);

#include "batcher.h"
// The RK4 forward kernel fits (a plan may hold only the Q2 layout).
bool onchip_forward_ok(const OnchipPlan* oc);
// Element-wise FP64 -> FP32 copy (tables for the mixed-precision adjoint).
void onchip_to_f32(const double* src, float* dst, long long n, cudaStream_t st);
bool onchip_mixed(const OnchipPlan* oc);
// acc += sums in block order: of gF_cta over ngF blocks, of acc_cta over nblk blocks.
void onchip_reduce(const OnchipPlan* oc, const double* gF_cta, int ngF, const double* acc_cta, int nblk, long long nst,
                   int K, int n1, int ne, GradAcc acc, cudaStream_t st);

// Suzuki-Trotter evolution (Sec. 2.3, App. A) of N Q2 sub-steps, lab frame, from psi_in
// to psi_out (API layout, may alias).  rows: (N + 1) x nq x d^2 1-body unitaries of the
// stage precision (row N = the first half of sub-step 0; row n = the last half of
// sub-step n followed by the first of sub-step n + 1); edges: per set s < nset and
// coupling e the half-step and full-step d^2 x d^2 unitaries at matrix (s ne + e) 2 + {0, 1};
// sub-step n uses set set_of[n % J].  q1: the first-order product instead (per step the
// couplings once each with their full-step unitary, then the next step's full-step
// 1-body row).  SG_E_UNSUPPORTED beyond 16 modes or 32 couplings.
sg_status onchip_q2_forward(const OnchipPlan* oc, const KPlan& p, const void* rows, const void* edges,
                            const double2* psi_in, double2* psi_out, int N, int J, const int* set_of, int nset,
                            cudaStream_t st, int* launches, bool q1 = false);
int onchip_dl(const OnchipPlan* oc);
// Suzuki-Trotter pulse gradient: pulls the final states psi and the co-state bar (API
// layout, lab frame) back through every factor of the N Q2 sub-steps and adds dF/df_k
// at sub-step n to gF_cta (CTA-major blocks of nstK >= N K doubles, slot n K + k;
// zeroed by the caller).  rows: [N][2 nq + K][d^2], per sub-step the inverse 1-body
// half-step factors U_i(n)^-1 (states), their adjoints U_i(n)^dag (co-states), then
// M_k(n) = U_i(n)^-1 L_k(n) with L_k the Frechet derivative of the local exponential
// along drive k's operator; edges: per set and coupling the inverse (half, full) and
// adjoint (half, full) coupling factors.  q1: the first-order product (N steps, rows of
// its full-step factors; the couplings pulled back in reverse order by their full-step
// factors).  SG_E_UNSUPPORTED for one mode, more than 32 couplings or 16 drives, or when
// the layout does not fit in shared memory.
sg_status onchip_q2_pulse_adjoint(const OnchipPlan* oc, const KPlan& p, const int* drv_mode, int K, const void* rows,
                                  const void* edges, const double2* psi, const double2* bar, int N, int J,
                                  const int* set_of, int nset, long long nstK, double* gF_cta, cudaStream_t st,
                                  int* launches, bool q1 = false);

// On-chip RK4 kernels for Hamiltonians that are real up to the frame phases (see
// onchip_real.cu): every mode has the same level count, every operator is parity-odd and
// real, or imaginary on both sides of a coupling, and the frame is the interaction picture.
#pragma once
#include <vector>
#include "kplan.h"
#include "grad.cuh"

// What the kernels need to know about the terms beyond the Kronecker-sum plan.
struct OcrTerms {
  int K = 0, sumd = 0;
  int eoff[SG_MAXQ] = {0}, opd_off[SG_MAXQ] = {0};   // offsets of a mode's levels and operators
  int drv_start[SG_MAXQ + 1] = {0}, drv_list[SG_MAXDRIVE] = {0};   // drives of each 1-body slot
  int drv_op[SG_MAXDRIVE] = {0};
  int e_opa[SG_MAXEDGE] = {0}, e_opb[SG_MAXEDGE] = {0};
  // Which part of an operator holds its real matrix (0 real, 1 imaginary), per coupling side,
  // and the modes whose basis is turned by i on odd levels: a parity-odd operator then changes
  // its part, so that drives are real and the two factors of a coupling alike (a drive's
  // part is its mode's flip).
  int e_pa[SG_MAXEDGE] = {0}, e_pb[SG_MAXEDGE] = {0};
  unsigned flip = 0;
};

struct OcrPlan;   // opaque
// nullptr when the plan is not one of these (2..6 modes, operators parity-odd, the
// couplings routable, shared memory); cols: columns of a state image, padding included.
OcrPlan* ocr_plan_create(const KPlan& p, bool mixed, const OcrTerms& t, int cols);
void ocr_plan_destroy(OcrPlan* o);
int ocr_ctas(const OcrPlan* o);
int ocr_resident(const OcrPlan* o);          // CTAs of the forward launch that one SM holds
void ocr_signature(const OcrPlan* o, std::vector<long long>& sig);
// The frame phases of half a step, exp(-i E dt/2) per composite level (D entries of the
// stage precision).
void ocr_half_step(const OcrPlan* o, const double* E, double dt, void* q, cudaStream_t st);

// Gradient: the forward and pull-back launches store their stage inputs (images [4 (step -
// n0) + stage][column][D]); one launch contracts the cross-densities of steps n0 .. n1 - 1:
// dF/df_k into gF (a block of nstK per column group, one store per stage slot) and, with ham,
// the term co-gradients into acc (ocr_blocks blocks of the GradAcc layout, added to).
bool ocr_adjoint_ok(const OcrPlan* o);
int ocr_blocks(const OcrPlan* o);
int ocr_groups(const OcrPlan* o);
int ocr_densities(const OcrPlan* o, const void* u, const void* k, const void* coef, const double2* opd, const double* J,
                  int n0, int n1, double dt, bool ham, long long nstK, double* gF, double* acc, cudaStream_t st);

// Many systems of one structure from their own start columns (FP32, one chunk each): per
// system the flat operators and couplings, the coefficients (3N x K), the frame phases of
// every step's middle (N x sumd), the half-step phases (D) and the columns (D x S, in and out).
struct OcrMany {
  const double2* opd;
  const double* J;
  const float* coef;
  const float2 *ph, *half;
  double2* psi;
  long long opd_n, J_n;           // entries per system
};
// Bytes of the device array that ocr_many fills with the systems' descriptions.
size_t ocr_many_bytes(int nsys);
cudaError_t ocr_many(const OcrPlan* o, const OcrMany& m, int nsys, int N, double dt, void* table, cudaStream_t st);

struct OcBatch;
int ocr_forward(const OcrPlan* o, OcBatch& bt, double dt, cudaStream_t st);

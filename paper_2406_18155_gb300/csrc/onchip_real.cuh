// Kernels of onchip_real.h, instantiated for FP32 (mixed) and FP64 in files of their own.
// On-chip RK4 with real operators.
//
// In the interaction picture H_I(t) = P(t) H(t) P(t)^dag with P = diag exp(i E t) and
// H(t) = sum_k f_k(t) O_k + sum_e J_e A_e (x) B_e, whose matrices are real and constant (a
// coupling of two imaginary factors is -J Im A (x) Im B; where a real factor meets an imaginary
// one, as a transmon's charge and a fluxonium's, turning the odd levels of one mode by i makes
// them alike, OcrTerms::flip).  The complex-row kernels
// (onchip.cu) form every matrix of H_I(t) per stage and multiply complex by complex.  Here
// the stage inputs are kept as u = P(t)^dag y: between two half steps P changes by the constant
// diagonal Q = exp(-i E h/2), so one RK4 step from psi (interaction picture, P_m = P at the
// step's middle) reads
//   b = P_m^dag psi
//   k1 = -i H(t) u,        u  = Q^dag b
//   k2 = -i H(t + h/2) u,  u  = b + h/2 q1,      q1 = Q k1
//   k3 = -i H(t + h/2) u,  u  = b + h/2 k2
//   k4 = -i H(t + h) u,    u  = Q (b + h k3)
//   psi += h/6 P_m (q1 + 2 k2 + 2 k3 + Q^dag k4)
// which is the interaction-picture RK4 step up to rounding.  The co-state lambda is pulled
// back by the same loop, steps and stage rows in reverse order, with v = i H kappa for k:
//   b = P_m^dag lambda
//   kappa4 = Q h/6 b                  v4 = i H(t + h) kappa4,     w4 = Q^dag v4
//   kappa3 = h/3 b + h w4             v3 = i H(t + h/2) kappa3
//   kappa2 = h/3 b + h/2 v3           v2 = i H(t + h/2) kappa2
//   kappa1 = Q^dag (h/6 b + h/2 v2)   v1 = i H(t) kappa1
//   lambda += P_m (w4 + v3 + v2 + Q v1)
// (the discrete adjoint of the step; with Q^dag stored for Q the two loops differ in
// constants only).
//
// What is constant for a whole solve must not be rounded to FP32: its error has one direction in
// every step (fl(h/6) is low by 4.5e-8 at h = 0.01, and so was every increment).  So
// H enters as G = h/6 H, formed in FP64 before it is rounded, and kappa as 6/h kappa: the weights
// above become 1, 2, 3 and 6 (the densities give back h/6).  Q is rounded to a number of
// modulus 1 (unit_phase32): an error of its angle turns the terms of stages 1 and 4 by
// opposite angles, which cancel from step to step, an error of its modulus does not.  The phases
// P_m, which turn the state and its increment back, have modulus 1 on average (unit_cis32).
// Against 64 bits, D = 25 pair, 10,000 steps, worst of five inputs: pulse gradient 5.5e-7 -> 1.5e-7
// (complex rows 6.5e-7), Hamiltonian gradient 9.6e-7 -> 2.8e-7 (2.1e-6); five modes of four levels, 2560
// steps: state 1.2e-7 -> 9e-8; at the same speed (1.57 ms, 6-mode chain 106 ms).
//
// psi stays in the interaction picture, so no phase error accumulates in it: P_m is read from the
// phase table every step.  Real times complex halves the multiply-adds (one packed FP32x2 FMA
// each), and the matrices stay in shared memory for the whole run; a stage reads K drive coefficients
// from memory instead of a row of term matrices.
//
// Work split.  A thread owns one d x d block over two modes at a time.  The modes are
// taken in pairs, one phase per pair (an odd last mode shares its partner), instead of one
// phase per coupling: a coupling between two phases is passed on as an image, w = B u
// written by the phase that holds B's mode and multiplied by J A in the phase that holds A's
// mode.  So a 6-mode chain takes 3 phases and 11 image accesses of an entry per stage where
// the phase-per-coupling form takes 5 phases and 23, and a pair of modes needs no exchange at
// all.  The last phase's blocks keep b, the increment and Q in registers (FP64 and d = 5: in
// shared memory, one column per thread), and the state as a float-float pair in shared
// memory, touched once per step.
//
// Measured, complex rows -> this: six fluxoniums (D = 4096, 64 columns, one CTA of 8 warps each)
// 35.5 -> 17.5 us a step, 1,450 instructions per warp and stage, 31 % of the issue slots (two warps
// per scheduler: fixed latencies and shared-memory waits); five modes of five levels (D = 3125, 4
// warps a column) 34.6 -> 26 us; gradient of the D = 25 pair, 10,000 mixed steps in 910 chunks,
// 1.42 ms of pull-back with densities -> 0.16 + 0.10 ms.
#pragma once
#include <algorithm>
#include <cstdint>
#include <vector>
#include "sg_internal.h"
#include "slab.h"
#include "slab_dev.cuh"
#include "onchip_dev.cuh"
#include "onchip_real.h"

constexpr int kRMat = 24;         // constant matrices of a plan
constexpr int kROne = 3;          // one-body matrix elements a thread renews per stage
constexpr int kRBuf = 2;          // exchange images beside u and the running sum
constexpr int kRImp = 3;          // images a phase reads

// Stored row length: the most nonzeros of a row.
__host__ __device__ constexpr int zrow(int DL) { return (DL + 1) / 2; }

// Where the blocks of the kernels for NQ modes of DL levels lie: all strides are compile-time
// constants, so a block's accesses are immediate offsets of one address per phase.  Phases
// take the modes in pairs, an odd last mode with its predecessor.
template <int DL, int NQ>
struct Lay {
  __host__ __device__ static constexpr int st(int k) {            // API stride of mode k
    int s = 1;
    for (int i = k; i < NQ - 1; ++i) s *= DL;
    return s;
  }
  __host__ __device__ static constexpr int pad(int x) { return DL == 2 || DL == 4 ? x + (x >> 4) + (x >> 8) : x; }
  static constexpr int NP = (NQ + 1) / 2;
  static constexpr int NBC = st(1);                               // blocks of a column (D / DL^2)
  static constexpr int SC = NBC >= 32 ? 1 : 32 / NBC;             // columns of a CTA, at most
  static constexpr int NT = (SC * NBC + 31) / 32 * 32;            // threads
  static constexpr int CS = (pad(st(0) * DL - 1) + 2) / 2 * 2;    // column stride of an image
  static constexpr int IMG = SC * CS;
  __host__ __device__ static constexpr int mode_a(int p) { return 2 * p < NQ - 2 ? 2 * p : NQ - 2; }
  // the other modes in thread order: the lowest even power of DL, the lowest odd one, then
  // the rest upwards (a half-warp's accesses then fall on different banks, slab_dev.cuh)
  __host__ __device__ static constexpr int other(int p, int j) {
    int ord[NQ] = {}, n = 0;
    const int a = mode_a(p), b = a + 1;
    for (int par = 0; par < 2; ++par)
      for (int k = NQ - 1; k >= 0; --k)
        if (k != a && k != b && (NQ - 1 - k) % 2 == par) { ord[n++] = k; break; }
    for (int k = NQ - 1; k >= 0; --k) {
      bool used = k == a || k == b;
      for (int i = 0; i < n; ++i) used = used || ord[i] == k;
      if (!used) ord[n++] = k;
    }
    return ord[j];
  }
};

// One pair of modes (a, b); matrix slots are -1 where absent.
struct OcrPhase {
  int mR, mL, expR;               // t = R u on b; sum += L t on a; t kept in image expR
  int mR2, mL2;                   // a second coupling of the pair
  int mE, expL;                   // image expL = E u on a
  int bA, bB;                     // one-body slots of a and b
  int nimp, imp_buf[kRImp], imp_mat[kRImp], imp_a[kRImp];   // sum += M (image) on a (1) or b (0)
};

struct OcrArgs {
  int D, S, cols, Sc, nbc, ncta, np, nbuf;
  int K, sumd, sumdA, n1, nmat;
  OcrPhase ph[3];
  int eoff[SG_MAXQ];              // level offsets of the modes in a phase row
  unsigned flip;                  // modes whose odd levels are turned by i
  // constant matrices: element (x, c) is part of opd[off + x d + c], times sign, times J
  int m_off[kRMat], m_part[kRMat], m_flip[kRMat], m_sign[kRMat], m_J[kRMat];
  // one-body slots: drives and their operators
  int d_start[SG_MAXQ + 1], d_drv[SG_MAXDRIVE], d_off[SG_MAXDRIVE], d_flip[SG_MAXQ];
  // shared-memory byte offsets
  int s_img, s_psi, s_b, s_acc, s_Q, s_mat, s_one, s_ph;
};

constexpr int kRSlot = 16;        // slots per CTA (warps)
constexpr int kDensFlush = 64;    // images between moves of the sums to FP64
struct OcdSlot {
  int kind;                       // 0 one-body, 1 side of a coupling
  int drv, mslot, edge, side;     // kind 0: drive and 1-body slot; kind 1: coupling and side
  int off, part, flip, sign;      // the slot's own operator: opd offset, part; sign of i A (x) i B
  int mat;                        // kind 1: the other factor's matrix (J included on side 1)
  int s1, s2;                     // image strides of the slot's digit and of its partner
  int no, pst[4];
};
struct OcdArgs {
  int D, cols, Cg, ncg, nbc, CS, K, sumd, n1, ne, ham;
  int nslot, nmat, ni;            // slots; matrices; images per load (1, or whole steps)
  long long accd, nstK;
  OcdSlot slot[kRSlot];
  int m_off[kRMat], m_part[kRMat], m_flip[kRMat], m_sign[kRMat], m_J[kRMat];
  int s_img, s_mat, s_g;
};
struct OcdJob {
  const void *u, *k, *coef;
  const double2* opd;
  const double* J;
  double *gF, *acc;
  int n0, n1;
  double dt;
};

struct HalfArgs {
  int D, nq, DL;
  int eoff[SG_MAXQ];
  double dt;
  const double* E;
};
struct OcrPlan {
  OcrArgs a{};
  OcdArgs dens{};                 // cross-densities: drives first, then the couplings' sides
  int dgrid = 1, ndrv = 0;        // CTAs along the steps; drive slots
  bool dens_ok = false;
  size_t dsmem = 0;
  HalfArgs half{};
  bool mixed = false;
  int DL = 0, nq = 0;
  size_t smem = 0;
};


// Launches of one precision (onchip_real_f32.cu, onchip_real_f64.cu).
// forward: bt null asks for the CTAs that an SM holds.
int ocr_fwd_f32(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st);
int ocr_fwd_f64(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st);
int ocr_dens_f32(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st);
int ocr_dens_f64(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st);

#ifdef OCR_KERNELS
namespace {

// the columns of row x that a parity-odd matrix keeps: c = zc(x, 0 .. zn(x) - 1)
template <int DL> __host__ __device__ constexpr int zn(int x) { return x & 1 ? (DL + 1) / 2 : DL / 2; }
__host__ __device__ constexpr int zc(int x, int j) { return 2 * j + (x & 1 ? 0 : 1); }

// The real matrix element in row x of an operator whose `part` holds it, in a basis turned by
// g = i on the odd levels (flip): conj(g_x) X_xc g_c for a parity-odd X = m or i m.
__device__ __forceinline__ double r_sign(int part, int flip, int x) { return flip && ((x & 1) ^ part) ? -1.0 : 1.0; }
__device__ __forceinline__ double r_elem(double2 o, int part, int flip, int x) {
  return r_sign(part, flip, x) * (part ? o.y : o.x);
}

__device__ __forceinline__ float2 zdup(float v) { return make_float2(v, v); }
__device__ __forceinline__ double zdup(double v) { return v; }

// o += M y along the block's first (LEFT) or second digit
template <int DL, bool LEFT, typename Z, typename C>
__device__ __forceinline__ void z_acc(const Z* __restrict__ M, const C (&y)[DL][DL], C (&o)[DL][DL]) {
#pragma unroll
  for (int x = 0; x < DL; ++x)
#pragma unroll
    for (int j = 0; j < zn<DL>(x); ++j) {
      const Z m = M[x * zrow(DL) + j];
#pragma unroll
      for (int z = 0; z < DL; ++z) {
        if (LEFT) o[x][z] = zfma(m, y[zc(x, j)][z], o[x][z]);
        else o[z][x] = zfma(m, y[z][zc(x, j)], o[z][x]);
      }
    }
}

// o += this phase's terms on the block u; img: the thread's place in the images (u, the
// running sum, then the exchange images, IMG entries apart).
template <int DL, int NQ, int P, typename Z, typename C>
__device__ __forceinline__ void z_phase(const OcrPhase& ph, const Z* __restrict__ mat, const Z* __restrict__ one,
                                        const C (&u)[DL][DL], C (&o)[DL][DL], C* img) {
  typedef Lay<DL, NQ> Y;
  constexpr int MS = DL * zrow(DL), SA = Y::pad(Y::st(Y::mode_a(P))), SB = Y::pad(Y::st(Y::mode_a(P) + 1));
  constexpr bool EX = Y::NP > 1;
  if (EX) {
#pragma unroll 1
    for (int i = 0; i < ph.nimp; ++i) {
      const C* w = img + (2 + ph.imp_buf[i]) * Y::IMG;
      const Z* M = mat + ph.imp_mat[i] * MS;
      C v[DL][DL];
#pragma unroll
      for (int x = 0; x < DL; ++x)
#pragma unroll
        for (int z = 0; z < DL; ++z) v[x][z] = w[x * SA + z * SB];
      if (ph.imp_a[i]) z_acc<DL, true>(M, v, o);
      else z_acc<DL, false>(M, v, o);
    }
  }
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
    const int mR = r ? ph.mR2 : ph.mR, mL = r ? ph.mL2 : ph.mL;
    if (mR < 0) break;
    C t[DL][DL];
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int z = 0; z < DL; ++z) t[x][z] = cmk<C>(0.0, 0.0);
    z_acc<DL, false>(mat + mR * MS, u, t);
    if (EX && r == 0 && ph.expR >= 0) {
      C* w = img + (2 + ph.expR) * Y::IMG;
#pragma unroll
      for (int x = 0; x < DL; ++x)
#pragma unroll
        for (int z = 0; z < DL; ++z) w[x * SA + z * SB] = t[x][z];
    }
    if (mL >= 0) z_acc<DL, true>(mat + mL * MS, t, o);
  }
  if (EX && ph.mE >= 0) {
    C* w = img + (2 + ph.expL) * Y::IMG;
    C t[DL][DL];
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int z = 0; z < DL; ++z) t[x][z] = cmk<C>(0.0, 0.0);
    z_acc<DL, true>(mat + ph.mE * MS, u, t);
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int z = 0; z < DL; ++z) w[x * SA + z * SB] = t[x][z];
  }
  if (ph.bA >= 0) z_acc<DL, true>(one + ph.bA * MS, u, o);
  if (ph.bB >= 0) z_acc<DL, false>(one + ph.bB * MS, u, o);
}

// Phase P of a stage: u from its image, the running sum from and to its own.
template <int DL, int NQ, int P, typename Z, typename C>
__device__ __forceinline__ void z_stage(const OcrArgs& a, const Z* __restrict__ mat, const Z* __restrict__ one,
                                        C (&u)[DL][DL], C (&o)[DL][DL], C* img) {
  typedef Lay<DL, NQ> Y;
  constexpr int SA = Y::pad(Y::st(Y::mode_a(P))), SB = Y::pad(Y::st(Y::mode_a(P) + 1));
#pragma unroll
  for (int x = 0; x < DL; ++x)
#pragma unroll
    for (int z = 0; z < DL; ++z) {
      if (Y::NP > 1) u[x][z] = img[x * SA + z * SB];
      o[x][z] = P ? img[Y::IMG + x * SA + z * SB] : cmk<C>(0.0, 0.0);
    }
  z_phase<DL, NQ, P>(a.ph[P], mat, one, u, o, img);
  if (P + 1 < Y::NP) {
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int z = 0; z < DL; ++z) img[Y::IMG + x * SA + z * SB] = o[x][z];
  }
}

template <typename R> struct Regs { __host__ __device__ static constexpr bool of(int DL) { return sizeof(R) == 4 && DL <= 4; } };

// A block of values that a thread keeps for itself: registers, or its own places of
// shared memory (entry-major, so a warp's accesses are consecutive).
template <bool REG, int N, typename C> struct Own;
template <int N, typename C> struct Own<true, N, C> {
  C r[N];
  __device__ void init(unsigned char*, int, int) {}
  __device__ __forceinline__ C get(int e) const { return r[e]; }
  __device__ __forceinline__ void set(int e, C v) { r[e] = v; }
};
template <int N, typename C> struct Own<false, N, C> {
  C* p;
  int st;
  __device__ void init(unsigned char* base, int tid, int stride) { p = reinterpret_cast<C*>(base) + tid; st = stride; }
  __device__ __forceinline__ C get(int e) const { return p[e * st]; }
  __device__ __forceinline__ void set(int e, C v) { p[e * st] = v; }
};

// One-body matrices of stage row q into `one`: sum over the slot's drives of f_k O_k.  The
// first drive's coefficient comes from f0 (loaded a stage ahead).  An element enters as its
// rounding and the remainder (f h + f l): an element rounded alone is a constant error of H that
// adds up over the steps, where the product's rounding changes with f.  Against FP64 over 6000
// steps of a 6-mode chain, largest gradient error over the largest component, with the constants of
// the step as above: 1.3e-4 (rounded alone 1.1e-3, complex-row kernels 7.6e-4).
template <typename R> struct OpEl {
  R h = 0, l = 0;
  OpEl() = default;
  __device__ __forceinline__ explicit OpEl(double o) : h((R)o), l((R)(o - (double)(R)o)) {}
  __device__ __forceinline__ R times(R f, R acc) const { return fma(f, h, fma(f, l, acc)); }
};
template <int DL, typename R, typename Z>
__device__ __forceinline__ void one_body(const OcrArgs& a, const R* __restrict__ coef, const double2* __restrict__ opd,
                                         double hs, int q, int i, R f0, OpEl<R> o0, Z* one) {
  constexpr int MS = DL * zrow(DL);
  const int u = i / MS, r = i - u * MS, x = r / zrow(DL), j = r - x * zrow(DL);
  R v = o0.times(f0, (R)0);
  if (j < zn<DL>(x))
    for (int k = a.d_start[u] + 1; k < a.d_start[u + 1]; ++k)
      v = OpEl<R>(hs * r_elem(opd[a.d_off[k] + x * DL + zc(x, j)], a.d_flip[u], a.d_flip[u], x))
              .times(coef[(size_t)q * a.K + a.d_drv[k]], v);
  one[i] = zdup(v);
}

template <typename R, int DL, int NQ>
__global__ void __launch_bounds__((Lay<DL, NQ>::NT), 1)
k_ocr_fwd(const __grid_constant__ OcrArgs a, double dt, const __grid_constant__ OcBatch bt) {
  typedef typename CT<R>::T C;
  typedef typename ZM<R>::T Z;
  constexpr int DD = DL * DL, MS = DL * zrow(DL);
  constexpr bool REG = Regs<R>::of(DL);
  typedef Lay<DL, NQ> Y;
  constexpr int NP = Y::NP, nthr = Y::NT, NO = NQ - 2;
  constexpr int MA = Y::mode_a(NP - 1), STA = Y::st(MA), STB = Y::st(MA + 1);    // the last phase's modes
  constexpr int SA = Y::pad(STA), SB = Y::pad(STB);
  extern __shared__ __align__(16) unsigned char sm[];
  int chunk, cta;
  const OcSys& d = oc_locate(bt, a.ncta, chunk, cta);
  const int tid = threadIdx.x;
  const int n0 = d.n0 + chunk * d.L, nsteps = min(d.n1, n0 + d.L) - n0, rev = d.rev;
  const R* __restrict__ coef = static_cast<const R*>(d.coef);
  const C* __restrict__ ph = static_cast<const C*>(d.ph);
  // H enters as G = h/6 H; epilogue constants (see the top): u' = c1 b + c2 k after stages 0, 1, 2 (2:
  // times Q), the increment acc + Q^dag k, k = -i G u with weight wk; rev: k = i G kappa
  const double hs = dt / 6;
  const R sg = rev ? (R)-1 : (R)1, wk = rev ? (R)1 : (R)2, c1a = rev ? (R)2 : (R)1, c2a = rev ? (R)6 : (R)3;
  const R c2c = rev ? (R)3 : (R)6;
  C* const img = d.segY ? static_cast<C*>(d.segY) + (size_t)4 * chunk * d.L * a.cols * a.D : nullptr;
  C* const us = reinterpret_cast<C*>(sm + a.s_img);
  Z* const mat = reinterpret_cast<Z*>(sm + a.s_mat);
  Z* const one = reinterpret_cast<Z*>(sm + a.s_one);
  C* const phs = reinterpret_cast<C*>(sm + a.s_ph);
  // this thread's column and blocks
  const int c = tid / Y::NBC, blk = tid - c * Y::NBC, col = cta * a.Sc + c;
  const bool on = c < a.Sc && col < a.cols;
  C* at[NP];                                        // its places in the u image, phase by phase
  int t0 = 0, dig[NO > 0 ? NO : 1];                 // API row and other digits of the last phase's block
  {
    int b[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      b[p] = blk;
      at[p] = us + (on ? c * Y::CS : 0);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int j = 0; j < NO; ++j) {
        const int x = b[p] % DL;
        b[p] /= DL;
        at[p] += x * Y::pad(Y::st(Y::other(p, j)));
        if (p == NP - 1) {
          dig[j] = x;
          t0 += x * Y::st(Y::other(p, j));
        }
      }
  }
  StateArr<R> ps;
  {
    unsigned char* base = sm + a.s_psi;
    if constexpr (sizeof(R) == 4) {
      ps.h = reinterpret_cast<float2*>(base) + tid;
      ps.l = ps.h + DD * nthr;
    } else {
      ps.p = reinterpret_cast<double2*>(base) + tid;
    }
  }
  Own<REG, DD, C> bv, acc, Q;
  bv.init(sm + a.s_b, tid, nthr);
  acc.init(sm + a.s_acc, tid, nthr);
  Q.init(sm + a.s_Q, tid, nthr);
  // constant matrices
  for (int i = tid; i < a.nmat * MS; i += nthr) {
    const int m = i / MS, r = i - m * MS, x = r / zrow(DL), j = r - x * zrow(DL);
    double v = 0.0;
    if (j < zn<DL>(x)) {
      const double2 o = d.opd64[a.m_off[m] + x * DL + zc(x, j)];
      v = r_elem(o, a.m_part[m], a.m_flip[m], x);
      if (a.m_J[m] >= 0) v *= d.J[a.m_J[m]] * a.m_sign[m] * hs;
    }
    mat[i] = zdup((R)v);
  }
  // one-body elements that this thread keeps up to date (the plan has at most kROne a thread)
  const int nB = a.n1 * MS;
  OpEl<R> o0[kROne];
  R f0[kROne];
  int k0[kROne];
#pragma unroll
  for (int e = 0; e < kROne; ++e) {
    const int i = tid + e * nthr;
    f0[e] = 0;
    k0[e] = -1;
    if (i < nB) {
      const int u = i / MS, r = i - u * MS, x = r / zrow(DL), j = r - x * zrow(DL);
      const int k = a.d_start[u];
      if (k < a.d_start[u + 1] && j < zn<DL>(x)) {
        k0[e] = a.d_drv[k];
        o0[e] = OpEl<R>(hs * r_elem(d.opd64[a.d_off[k] + x * DL + zc(x, j)], a.d_flip[u], a.d_flip[u], x));
      }
    }
  }
  // table row of stage s of the i-th step taken
  auto row_of = [&](int i, int s) {
    return rev ? 3 * (n0 + nsteps - 1 - i) + 2 - stage_row(s) : 3 * (n0 + i) + stage_row(s);
  };
  auto load_f = [&](int q) {
#pragma unroll
    for (int e = 0; e < kROne; ++e)
      if (k0[e] >= 0) f0[e] = coef[(size_t)q * a.K + k0[e]];
  };
  auto store_one = [&](int q, Z* to) {
#pragma unroll
    for (int e = 0; e < kROne; ++e) {
      const int i = tid + e * nthr;
      if (i < nB) one_body<DL, R>(a, coef, d.opd64, hs, q, i, f0[e], o0[e], to);
    }
  };
  auto mid_phases = [&](int i, C* to) {            // the phases of step i's middle, by cp.async
    const int q = row_of(i, 1);
    const C* src = ph + (size_t)(d.phmid ? q / 3 : q) * a.sumd;
    for (int j = tid; j < a.sumd; j += nthr) cpv(to + j, src + j);
  };
  if (on) {
#pragma unroll
    for (int e = 0; e < DD; ++e) {
      const int t = t0 + e / DL * STA + e % DL * STB;
      double2 v = make_double2(0.0, 0.0);
      if (d.img_in) v = d.img_in[((size_t)chunk * a.cols + col) * a.D + t];
      else if (d.ident) v.x = col == t ? 1.0 : 0.0;
      else if (col < a.S) v = d.psi_api[(size_t)t * a.S + col];
      ps.set(e * nthr, v);
      C q = static_cast<const C*>(d.half)[t];
      if (rev) q.y = -q.y;
      Q.set(e, q);
    }
  }
  // P at the step's middle for this thread's block: (product over the other modes) x first digit,
  // times second digit
  auto phases = [&](const C* row, C (&pa)[DL]) {
    C f = cmk<C>(1.0, 0.0);
#pragma unroll
    for (int j = 0; j < NO; ++j) {
      f = cmulT(f, row[a.eoff[Y::other(NP - 1, j)] + dig[j]]);
      if (((a.flip >> Y::other(NP - 1, j)) & 1u) && (dig[j] & 1)) f = cmk<C>(-f.y, f.x);
    }
#pragma unroll
    for (int x = 0; x < DL; ++x) {
      pa[x] = cmulT(f, row[a.eoff[MA] + x]);
      if ((x & 1) && ((a.flip >> MA) & 1u)) pa[x] = cmk<C>(-pa[x].y, pa[x].x);
    }
  };
  auto phase_b = [&](const C* row, int z) {
    const C p = row[a.eoff[MA + 1] + z];
    return (z & 1) && ((a.flip >> (MA + 1)) & 1u) ? cmk<C>(-p.y, p.x) : p;
  };
  C u[DL][DL];
  // b = P_m^dag psi, u = Q^dag b
  auto begin_step = [&](const C* row) {
    C pa[DL];
    phases(row, pa);
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int z = 0; z < DL; ++z) {
        const int e = x * DL + z;
        const C p = cmulT(pa[x], phase_b(row, z));
        const C b = cmulT(cconjT(p), ps.hi(e * nthr));
        bv.set(e, b);
        u[x][z] = cmulT(cconjT(Q.get(e)), b);
        if (NP > 1) at[NP - 1][x * SA + z * SB] = u[x][z];
      }
  };
  if (nsteps > 0) {
    mid_phases(0, phs);
    load_f(row_of(0, 0));
    store_one(row_of(0, 0), one);
  }
  cp_wait_all();
  __syncthreads();
  if (nsteps > 0 && on) begin_step(phs);
  if (NP > 1) __syncthreads();
  int buf = 0;
  for (int i = 0; i < nsteps; ++i) {
    const C* const prow = phs + (i & 1) * a.sumdA;
    C* const pnext = phs + ((i & 1) ^ 1) * a.sumdA;
    if (d.ck_out && on && (rev ? (i == 0 || (nsteps - i) % d.K == 0) : i % d.K == 0)) {
      double2* ck = d.ck_out + ((size_t)((rev ? nsteps - 1 - i : i) / d.K) * a.cols + col) * a.D;
#pragma unroll
      for (int e = 0; e < DD; ++e) ck[t0 + e / DL * STA + e % DL * STB] = ps.get(e * nthr);
    }
    if (i + 1 < nsteps) mid_phases(i + 1, pnext);
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      const Z* const oc = one + buf * nB;
      const int ni = s < 3 ? i : i + 1, ns = s < 3 ? s + 1 : 0;
      const bool more = ni < nsteps;
      const int qn = more ? row_of(ni, ns) : 0;
      if (more) load_f(qn);
      if (img) {
        // this stage's input, in API order (the images are read back whole)
        C* g = img + ((size_t)(4 * (rev ? nsteps - 1 - i : i) + (rev ? 3 - s : s)) * a.cols + cta * a.Sc) * a.D;
        if (NP > 1) {
          const int ncol = min(a.Sc, a.cols - cta * a.Sc);
          for (int e = tid; e < ncol * a.D; e += nthr) {
            const int cc = e / a.D, t = e - cc * a.D;
            g[e] = us[cc * Y::CS + spos<DL>(t)];
          }
        } else if (on) {
#pragma unroll
          for (int e = 0; e < DD; ++e) g[(size_t)c * a.D + t0 + e / DL * STA + e % DL * STB] = u[e / DL][e % DL];
        }
      }
      C o[DL][DL];
      if (on) z_stage<DL, NQ, 0>(a, mat, oc, u, o, at[0]);
      if constexpr (NP > 1) {
        __syncthreads();
        if (on) z_stage<DL, NQ, 1>(a, mat, oc, u, o, at[1]);
      }
      if constexpr (NP > 2) {
        __syncthreads();
        if (on) z_stage<DL, NQ, 2>(a, mat, oc, u, o, at[2]);
      }
      // (the inner stages share one loop: the code is larger than the instruction cache's reach)
      const R wks = s == 0 ? (R)1 : wk, c1s = s == 2 ? (R)1 : c1a, c2s = s == 0 ? c2a : s == 1 ? (R)3 : c2c;
      if (on) {
        // epilogue on the last phase's block
#pragma unroll
        for (int x = 0; x < DL; ++x)
#pragma unroll
          for (int z = 0; z < DL; ++z) {
            const int e = x * DL + z;
            C k = cmk<C>(sg * o[x][z].y, -sg * o[x][z].x);
            C v;
            if (s == 3) {
              const C g = acc.get(e), w = cmulT(cconjT(Q.get(e)), k);
              v = cmk<C>(g.x + w.x, g.y + w.y);
            } else {
              const C b = bv.get(e);
              C g = cmk<C>(0.0, 0.0);
              if (s == 0) k = cmulT(Q.get(e), k);
              else g = acc.get(e);
              acc.set(e, cmk<C>(g.x + wks * k.x, g.y + wks * k.y));
              v = cmk<C>(c1s * b.x + c2s * k.x, c1s * b.y + c2s * k.y);
              if (s == 2) v = cmulT(Q.get(e), v);
            }
            u[x][z] = v;
            if (NP > 1 && s < 3) at[NP - 1][x * SA + z * SB] = v;
          }
        if (s == 3) {
          C pa[DL];
          phases(prow, pa);
#pragma unroll
          for (int x = 0; x < DL; ++x)
#pragma unroll
            for (int z = 0; z < DL; ++z)
              ps.add((x * DL + z) * nthr, cmulT(cmulT(pa[x], phase_b(prow, z)), u[x][z]));
          if (i + 1 < nsteps) begin_step(pnext);
        }
      }
      if (more) store_one(qn, one + (buf ^ 1) * nB);
      cp_wait_all();
      __syncthreads();
      buf ^= 1;
    }
  }
  if (on) {
#pragma unroll
    for (int e = 0; e < DD; ++e) {
      const int t = t0 + e / DL * STA + e % DL * STB;
      const double2 v = ps.get(e * nthr);
      if (d.img_out) d.img_out[((size_t)chunk * a.cols + col) * a.D + t] = v;
      if (d.psi_out && col < a.S) d.psi_out[(size_t)t * a.S + col] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// cross-densities
// ---------------------------------------------------------------------------
// dF/dX of every term matrix X from the stored stage inputs u and kappa: with the other
// factor of the term applied, C_ab = sum conj(kappa_a) (u')_b over the slab, the frame phases
// cancel, and dF = sum_ab Im C_ab dX_ab (imaginary couplings: -Im C on their real matrices);
// the energies enter through P(t), t Re C_ab X_ab (grad.cuh).  The stages do not depend on one
// another, so this is one launch over all steps of a round, not a part of the serial
// pull-back.  X is constant, so a lane keeps its sums (weighted by f_k, and by t) in
// registers for all its steps and the warp adds them up once at the end; per stage only
// dF/df_k, one scalar per drive, is summed over the lanes.  One warp per slot (a drive, or a side
// of a coupling), lanes over the blocks of the slot's pair of modes; the images of the next
// steps arrive by cp.async meanwhile.  Bound by shared memory: 2 d^2 loads of 8 bytes per block
// against 2 to 3 d^3 multiply-adds.
template <int DL> __host__ __device__ constexpr int npair() { return DL * DL / 2; }

template <typename R, int DL>
__global__ void __launch_bounds__(32 * kRSlot, 1)
k_ocr_dens(const __grid_constant__ OcdArgs a, const __grid_constant__ OcdJob jb) {
  typedef typename CT<R>::T C;
  typedef typename ZM<R>::T Z;
  constexpr int MS = DL * zrow(DL), NPR = npair<DL>();
  extern __shared__ __align__(16) unsigned char sm[];
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, w = tid >> 5;
  const int cg = blockIdx.y, ncol = min(a.Cg, a.cols - cg * a.Cg);
  const int nst = jb.n1 - jb.n0;                         // this CTA's images: whole steps
  const int b0 = 4 * (int)((long long)nst * blockIdx.x / gridDim.x);
  const int b1 = 4 * (int)((long long)nst * (blockIdx.x + 1) / gridDim.x);
  const int imgn = a.Cg * a.CS;                          // entries of one image of the group
  C* const bufs = reinterpret_cast<C*>(sm + a.s_img);    // [2][u, kappa][ni images]
  Z* const mat = reinterpret_cast<Z*>(sm + a.s_mat);
  R* const gb = reinterpret_cast<R*>(sm + a.s_g) + w * 32;
  for (int i = tid; i < a.nmat * MS; i += nthr) {
    const int m = i / MS, r = i - m * MS, x = r / zrow(DL), j = r - x * zrow(DL);
    double v = 0.0;
    if (j < zn<DL>(x)) {
      const double2 o = jb.opd[a.m_off[m] + x * DL + zc(x, j)];
      v = r_elem(o, a.m_part[m], a.m_flip[m], x);
      if (a.m_J[m] >= 0) v *= jb.J[a.m_J[m]] * a.m_sign[m];
    }
    mat[i] = zdup((R)v);
  }
  const double hs = jb.dt / 6;                           // kappa comes as 6/h kappa
  const OcdSlot& S = a.slot[min(w, a.nslot - 1)];
  const bool on = w < a.nslot;
  // the slot's own operator (dF/df_k of a drive)
  R own[NPR];
  {
    int p = 0;
#pragma unroll
    for (int x = 0; x < DL; ++x)
#pragma unroll
      for (int j = 0; j < zn<DL>(x); ++j, ++p) {
        const double2 o = jb.opd[S.off + x * DL + zc(x, j)];
        own[p] = (R)r_elem(o, S.part, S.flip, x);
      }
  }
  R aI[NPR], aR[NPR];
#pragma unroll
  for (int p = 0; p < NPR; ++p) aI[p] = aR[p] = 0;
  // every kDensFlush images the warp's sums move to FP64, element p held by lane p (thousands of
  // FP32 additions to one sum would cost digits that the next sums cancel against; D = 3125, 1000
  // steps: error of the Hamiltonian gradient 5.5e-7 -> 1.8e-7)
  double kI = 0.0, kR = 0.0;
  int since = 0;
  auto flush = [&]() {
#pragma unroll
    for (int p = 0; p < NPR; ++p) {
      const double vI = warp_sum((double)aI[p]), vR = warp_sum((double)aR[p]);
      if (lane == p) { kI += vI; kR += vR; }
      aI[p] = aR[p] = 0;
    }
    since = 0;
  };
  const C* const gu = static_cast<const C*>(jb.u);
  const C* const gk = static_cast<const C*>(jb.k);
  const R* const coef = static_cast<const R*>(jb.coef);
  // images m, m + 1, ... of the launch into buffer b
  auto load = [&](int m, int b) {
    const int n = min(a.ni, b1 - m) * ncol * a.D;
    C* du = bufs + (size_t)b * 2 * a.ni * imgn;
    C* dk = du + a.ni * imgn;
    for (int e = tid; e < n; e += nthr) {
      const int im = e / (ncol * a.D), r = e - im * ncol * a.D, c = r / a.D, t = r - c * a.D;
      const size_t src = ((size_t)(m + im) * a.cols + cg * a.Cg + c) * a.D + t;
      const int dst = im * imgn + c * a.CS + spos<DL>(t);
      cpv(du + dst, gu + src);
      cpv(dk + dst, gk + src);
    }
  };
  if (b0 < b1) load(b0, 0);
  int buf = 0;
  const int items = ncol * a.nbc;                        // blocks of one image
  const bool big = items >= 32;
  double* const gF = jb.gF + (size_t)cg * a.nstK;
  R gmid = 0;                                            // stage 1's share of its slot 3n + 1
  for (int m = b0; m < b1; m += a.ni) {
    cp_wait_all();
    __syncthreads();
    if (m + a.ni < b1) load(m + a.ni, buf ^ 1);
    const int nim = min(a.ni, b1 - m);
    const C* const us = bufs + (size_t)buf * 2 * a.ni * imgn;
    const C* const kp = us + a.ni * imgn;
    if (on) {
      // one image at a time, or as many as fill the lanes
      const int per = big ? 1 : 32 / items;
      for (int im0 = 0; im0 < nim; im0 += per) {
        const int np = min(per, nim - im0);
        R g = 0;
        for (int it = lane; it < np * items; it += 32) {
          const int im = im0 + it / items, r = it % items, c = r / a.nbc;
          int b = r - c * a.nbc, at = im * imgn + c * a.CS;
          for (int j = 0; j < S.no; ++j) {
            at += b % DL * S.pst[j];
            b /= DL;
          }
          const int st = (m + im) & 3, n = jb.n0 + ((m + im) >> 2), q = 3 * n + stage_row(st);
          R cI[NPR], cR[NPR];
#pragma unroll
          for (int p = 0; p < NPR; ++p) cI[p] = cR[p] = 0;
          if (S.kind == 0) {
#pragma unroll
            for (int z = 0; z < DL; ++z) {
              C x[DL], y[DL];
#pragma unroll
              for (int i = 0; i < DL; ++i) {
                x[i] = kp[at + i * S.s1 + z * S.s2];
                y[i] = us[at + i * S.s1 + z * S.s2];
              }
              int p = 0;
#pragma unroll
              for (int i = 0; i < DL; ++i)
#pragma unroll
                for (int j = 0; j < zn<DL>(i); ++j, ++p) {
                  const C v = y[zc(i, j)];
                  cR[p] += x[i].x * v.x + x[i].y * v.y;
                  cI[p] += x[i].x * v.y - x[i].y * v.x;
                }
            }
          } else {
            const Z* M = mat + S.mat * MS;
            C y[DL][DL];
#pragma unroll
            for (int i = 0; i < DL; ++i)
#pragma unroll
              for (int z = 0; z < DL; ++z) y[i][z] = us[at + i * S.s1 + z * S.s2];
#pragma unroll
            for (int z = 0; z < DL; ++z) {
              C x[DL], t[DL];
#pragma unroll
              for (int i = 0; i < DL; ++i) {
                x[i] = kp[at + i * S.s1 + z * S.s2];
                t[i] = cmk<C>(0.0, 0.0);
              }
#pragma unroll
              for (int j = 0; j < zn<DL>(z); ++j) {
                const Z m = M[z * zrow(DL) + j];
#pragma unroll
                for (int i = 0; i < DL; ++i) t[i] = zfma(m, y[i][zc(z, j)], t[i]);
              }
              int p = 0;
#pragma unroll
              for (int i = 0; i < DL; ++i)
#pragma unroll
                for (int j = 0; j < zn<DL>(i); ++j, ++p) {
                  const C v = t[zc(i, j)];
                  cR[p] += x[i].x * v.x + x[i].y * v.y;
                  cI[p] += x[i].x * v.y - x[i].y * v.x;
                }
            }
          }
          const R f = S.kind == 0 ? coef[(size_t)q * a.K + S.drv] : (R)1;
          const R ft = f * (R)((double)(2 * n + stage_row(st)) * jb.dt * 0.5);
#pragma unroll
          for (int p = 0; p < NPR; ++p) {
            g += own[p] * cI[p];
            aI[p] += f * cI[p];
            aR[p] += ft * cR[p];
          }
        }
        if (S.kind == 0) {
          if (big) {
            g = warp_sum(g);
            const int st = (m + im0) & 3, q = 3 * (jb.n0 + ((m + im0) >> 2)) + stage_row(st);
            if (st == 1) gmid = g;
            else if (lane == 0) gF[(size_t)q * a.K + S.drv] = hs * (st == 2 ? (double)gmid + (double)g : (double)g);
          } else {
            // a lane per image: the sum of its items' shares in order
            gb[lane] = g;
            __syncwarp();
            R v = 0;
            if (lane < np)
              for (int r = 0; r < items; ++r) v += gb[lane * items + r];
            __syncwarp();
            gb[lane] = v;
            __syncwarp();
            if (lane < np) {
              const int im = m + im0 + lane, st = im & 3, q = 3 * (jb.n0 + (im >> 2)) + stage_row(st);
              double* const to = gF + (size_t)q * a.K + S.drv;
              // stages 1 and 2 share a slot: they are neighbours, in this pass or across two
              if (st == 0 || st == 3) *to = hs * (double)v;
              else if (st == 1 && lane + 1 < np) *to = hs * ((double)v + (double)gb[lane + 1]);
              else if (st == 1) *to = hs * (double)v;
              else if (lane == 0) *to += hs * (double)v;
            }
            __syncwarp();
          }
        }
      }
    }
    if (a.ham && (since += nim) >= kDensFlush) flush();
    __syncthreads();
    buf ^= 1;
  }
  if (!a.ham) return;
  flush();
  // the warp's sums, then lane 0 adds them to the CTA's block (GradAcc layout)
  double* const G = jb.acc + ((size_t)cg * gridDim.x + blockIdx.x) * a.accd;
  const int MD2 = SG_MAXD * SG_MAXD;
  double* const gD = G;
  double* const gL = gD + 2ll * a.K * MD2;
  double* const gR = gL + 2ll * a.ne * MD2;
  double* const geB = gR + 2ll * a.ne * MD2;
  double* const geL = geB + (long long)a.n1 * SG_MAXD;
  double* const geR = geL + (long long)a.ne * SG_MAXD;
  double* const gjb = geR + (long long)a.ne * SG_MAXD;
  const double Je = S.kind ? jb.J[S.edge] : 1.0;
  // side 0: C without J; the co-gradient of A and the energies take it, dF/dJ does not.  Side 1's matrix
  // carries J and the sign already.
  const double s1 = !S.kind || S.side ? 1.0 : Je * S.sign;
  double* const ob = S.kind == 0 ? gD + 2ll * S.drv * MD2 : (S.side ? gR : gL) + 2ll * S.edge * MD2;
  double* const eb = S.kind == 0 ? geB + S.mslot * SG_MAXD : (S.side ? geR : geL) + S.edge * SG_MAXD;
  // lane p has element p's sums; lane x gathers level x (one lane for all took 12 to 36 dependent
  // accesses to memory per slot, slot after slot: 0.2 ms of a launch)
  double eR = 0.0, dj = 0.0;
  int x = 0, y = 0;
  if (on && lane < NPR) {
    int r = lane;
    while (r >= zn<DL>(x)) r -= zn<DL>(x++);
    y = zc(x, r);
    const double m = r_elem(jb.opd[S.off + x * DL + y], S.part, S.flip, x);
    ob[2 * (x * SG_MAXD + y) + (S.part ? 1 : 0)] += r_sign(S.part, S.flip, x) * s1 * (hs * kI);
    eR = s1 * m * (hs * kR);
    dj = m * (hs * kI);
  }
  dj = warp_sum(dj);
  if (on && S.kind && S.side == 0 && lane == 0) gjb[S.edge] += S.sign * dj;
  double mine = 0.0;
  for (int l = 0; l < DL; ++l) {
    const double v = warp_sum(lane < NPR ? (x == l ? eR : 0.0) - (y == l ? eR : 0.0) : 0.0);
    if (lane == l) mine = v;
  }
  // one warp after the other: drives of one mode add to the same energies
  for (int turn = 0; turn < a.nslot; ++turn) {
    if (on && w == turn && lane < DL) eb[lane] += mine;
    __syncthreads();
  }
}


template <auto kern>
void ocr_smem_once() {
  static const bool done = [] {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
    return true;
  }();
  (void)done;
}

template <typename R, int DL, int NQ>
int ocr_t(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st) {
  // the states of these do not fit in shared memory (ocr_plan_create)
  if constexpr (DL == 5 && (NQ == 6 || (NQ == 5 && sizeof(R) == 8)) || DL == 4 && NQ == 6 && sizeof(R) == 8) {
    return 0;
  } else {
    ocr_smem_once<k_ocr_fwd<R, DL, NQ>>();
    if (!bt) {
      int n = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ocr_fwd<R, DL, NQ>, Lay<DL, NQ>::NT, o->smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
      }
      return n;
    }
    int g = 0;
    for (int b = 0; b < (bt->many ? 0 : bt->nsys); ++b) {
      bt->cta0[b] = g;
      g += bt->s[b].C * o->a.ncta;
    }
    if (bt->many) g = bt->nsys * bt->per;
    if (g > 0) k_ocr_fwd<R, DL, NQ><<<g, Lay<DL, NQ>::NT, o->smem, st>>>(o->a, dt, *bt);
    return 1;
  }
}

template <typename R, int DL>
int ocr_nq(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st) {
  switch (o->nq) {
    case 2: return ocr_t<R, DL, 2>(o, bt, dt, st);
    case 3: return ocr_t<R, DL, 3>(o, bt, dt, st);
    case 4: return ocr_t<R, DL, 4>(o, bt, dt, st);
    case 5: return ocr_t<R, DL, 5>(o, bt, dt, st);
    default: return ocr_t<R, DL, 6>(o, bt, dt, st);
  }
}

template <typename R>
int ocr_dl(const OcrPlan* o, OcBatch* bt, double dt, cudaStream_t st) {
  switch (o->DL) {
    case 2: return ocr_nq<R, 2>(o, bt, dt, st);
    case 3: return ocr_nq<R, 3>(o, bt, dt, st);
    case 4: return ocr_nq<R, 4>(o, bt, dt, st);
    default: return ocr_nq<R, 5>(o, bt, dt, st);
  }
}

template <typename R, int DL>
int dens_t(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st) {
  ocr_smem_once<k_ocr_dens<R, DL>>();
  k_ocr_dens<R, DL><<<dim3(o->dgrid, g.ncg), 32 * g.nslot, o->dsmem, st>>>(g, j);
  return 1;
}
template <typename R>
int dens_dl(const OcrPlan* o, const OcdArgs& g, const OcdJob& j, cudaStream_t st) {
  switch (o->DL) {
    case 2: return dens_t<R, 2>(o, g, j, st);
    case 3: return dens_t<R, 3>(o, g, j, st);
    case 4: return dens_t<R, 4>(o, g, j, st);
    default: return dens_t<R, 5>(o, g, j, st);
  }
}

}  // namespace
#endif

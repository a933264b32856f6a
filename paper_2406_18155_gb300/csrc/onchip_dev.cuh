// Device pieces shared by the on-chip evolution kernels (onchip.cu, onchip_real.cu):
// asynchronous copies, the float-float state, the description of a launch's solves.
#pragma once
#include <cstdint>
#include "kplan.h"

// One solve of a launch: its tables, buffers and chunks of steps.  A solve has C chunks
// of L steps, chunk c covering steps [n0 + c L, min(n1, n0 + (c + 1) L)), and every chunk
// has the plan's ncta CTAs; the CTAs of solve b of a launch start at cta0[b].
struct OcSys {
  const void* tab;
  const void* atab;      // adjoint: rows the co-state is pulled back with (tab: the forward
                         // rows, which the cross-densities contract)
  const void* coef;
  const void* ph;
  const void* opd;
  const double2* psi_api;
  const double2* img_in; // start images, one per chunk
  double2* img_out;      // forward: the chunks' final images
  double2* psi_out;
  double2* ck_out;
  void* segY;
  double2* pbar_img;     // adjoint: the co-states at the chunks' ends, one image per chunk
  double* gF_cta;
  double* acc_cta;
  int* err;
  void* pblo;
  const double* J;       // coupling strengths of the solve (device)
  const double2* opd64;  // real-operator kernels: truncated operators, FP64
  const void* half;      // and the frame phases of half a step
  int phmid;             // ph holds one row a step (its middle) instead of its three stages
  long long nstK;
  int n0, n1, K;
  int C, L;
  int ident;             // forward: column j starts in basis state j (a chunk's propagator)
  int rev;               // forward: the steps backwards (the co-state's pull-back, see k_oc_fwd)
};
constexpr int kOcMaxBatch = 24;
struct OcBatch {
  int nsys;
  int cta0[kOcMaxBatch];
  OcSys s[kOcMaxBatch];
  const OcSys* many;     // more solves than s holds: device array, `per` CTAs each
  int per;
};

namespace {

// ---------------------------------------------------------------------------
// asynchronous copies and barriers
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// cp.async of 4, 8 or 16 bytes global -> shared (no registers, completes at cp_wait_all)
__device__ __forceinline__ void cp4(void* s, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp8(void* s, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cpv(float2* s, const float2* g) { cp8(s, g); }
__device__ __forceinline__ void cpv(double2* s, const double2* g) { cp16(s, g); }
__device__ __forceinline__ void cpv(float* s, const float* g) { cp4(s, g); }
__device__ __forceinline__ void cpv(double* s, const double* g) { cp8(s, g); }

__device__ __forceinline__ void mb_init(uint64_t* mb) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(mb)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
// One bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) into
// shared memory, completing a phase of mb.  Issued by one thread.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* mb) {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(mb)), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(mb))
      : "memory");
}
__device__ __forceinline__ bool mb_try(uint64_t* mb, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(mb)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase `parity` of mb: true once the phase has completed,
// false after `limit` polls (about a second at the default limit).
__device__ __forceinline__ bool mb_wait_for(uint64_t* mb, unsigned parity, int limit) {
  for (int it = 0; it < limit; ++it) {
    if (mb_try(mb, parity)) return true;
    __nanosleep(64);
  }
  return false;
}
// Barrier among the first n threads of the CTA (n a multiple of 32); id 0 is __syncthreads.
__device__ __forceinline__ void bar_sub(int id, int n) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}

// ---------------------------------------------------------------------------
// state: complex128, or float-float pairs in mixed precision
// ---------------------------------------------------------------------------
// hi + lo <- hi + lo + x with hi = fl(hi + lo) afterwards (TwoSum, then a fast
// renormalisation); exact up to the rounding of the low word.
__device__ __forceinline__ void ff_add(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  const float e = (hi - (s - bb)) + (x - bb);
  const float l = lo + e;
  const float h2 = s + l;
  lo = l - (h2 - s);
  hi = h2;
}

template <typename R> struct StateArr;
template <> struct StateArr<double> {
  double2* p;
  __device__ void init(unsigned char* base, int n) { p = reinterpret_cast<double2*>(base); (void)n; }
  __device__ void set(int e, double2 v) { p[e] = v; }
  __device__ double2 get(int e) const { return p[e]; }
  __device__ double2 hi(int e) const { return p[e]; }
  __device__ void add(int e, double2 x) { p[e] = make_double2(p[e].x + x.x, p[e].y + x.y); }
};
template <> struct StateArr<float> {
  float2 *h, *l;
  __device__ void init(unsigned char* base, int n) {
    h = reinterpret_cast<float2*>(base);
    l = h + n;
  }
  // high words in shared memory, low words elsewhere (global memory when shared
  // memory is short: they are touched once per step)
  __device__ void init_split(unsigned char* base, float2* lo) {
    h = reinterpret_cast<float2*>(base);
    l = lo;
  }
  __device__ void set(int e, double2 v) {
    const float hx = __double2float_rn(v.x), hy = __double2float_rn(v.y);
    h[e] = make_float2(hx, hy);
    l[e] = make_float2(__double2float_rn(v.x - (double)hx), __double2float_rn(v.y - (double)hy));
  }
  __device__ double2 get(int e) const {
    return make_double2((double)h[e].x + (double)l[e].x, (double)h[e].y + (double)l[e].y);
  }
  __device__ float2 hi(int e) const { return h[e]; }
  __device__ void add(int e, float2 x) {
    float2 a = h[e], b = l[e];
    ff_add(a.x, b.x, x.x);
    ff_add(a.y, b.y, x.y);
    h[e] = a;
    l[e] = b;
  }
};

// The solve, chunk and CTA within the chunk that this block works on.
__device__ __forceinline__ const OcSys& oc_locate(const OcBatch& bt, int ncta, int& chunk, int& cta) {
  if (bt.many) {
    const int b = blockIdx.x / bt.per, rel = blockIdx.x - b * bt.per;
    chunk = rel / ncta;
    cta = rel - chunk * ncta;
    return bt.many[b];
  }
  int b = 0;
  while (b + 1 < bt.nsys && (int)blockIdx.x >= bt.cta0[b + 1]) ++b;
  const int rel = blockIdx.x - bt.cta0[b];
  chunk = rel / ncta;
  cta = rel - chunk * ncta;
  return bt.s[b];
}

template <typename V>
__device__ __forceinline__ void issue_rows(const V* __restrict__ tab, int row, int q, V* dst, int tid, int nthr) {
  const V* src = tab + (size_t)q * row;
  for (int i = tid; i < row; i += nthr) cpv(dst + i, src + i);
}

__host__ __device__ __forceinline__ int stage_row(int s) { return s == 0 ? 0 : (s == 3 ? 2 : 1); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename C> __device__ __forceinline__ C cmulT(C a, C b) {
  return cmk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cconjT(C a) { return cmk<C>(a.x, -a.y); }


}  // namespace

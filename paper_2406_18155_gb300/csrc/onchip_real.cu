// Real-operator on-chip solves: plans (how the terms are spread over the phases) and launches.
#include "onchip_real.cuh"
#include <cstring>
#include <type_traits>

namespace {

template <typename R>
__global__ void k_ocr_half(HalfArgs a, typename CT<R>::T* __restrict__ q) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < a.D; t += gridDim.x * blockDim.x) {
    double e = 0.0;
    int r = t;
    for (int i = a.nq - 1; i >= 0; --i) {
      e += a.E[a.eoff[i] + r % a.DL];
      r /= a.DL;
    }
    if constexpr (sizeof(R) == 4) {
      q[t] = unit_phase32(-0.5 * e * a.dt);
    } else {
      double sn, cs;
      sincos(-0.5 * e * a.dt, &sn, &cs);
      q[t] = make_double2(cs, sn);
    }
  }
}

size_t al16(size_t x) { return (x + 15) & ~size_t(15); }


}  // namespace

OcrPlan* ocr_plan_create(const KPlan& p, bool mixed, const OcrTerms& t, int cols) {
  const int nq = p.nq, DL = p.dims[0];
  if (nq < 2 || nq > 6 || DL < 2 || DL > 5 || p.D > 4096) return nullptr;
  long long s = 1;
  for (int i = nq - 1; i >= 0; --i) {
    if (p.dims[i] != DL || p.st[i] != s) return nullptr;
    s *= DL;
  }
  for (int u = 0; u < p.n1; ++u) if (!((p.par1 >> u) & 1u)) return nullptr;
  for (int e = 0; e < p.ne; ++e) if (!((p.parL >> e) & 1ull) || !((p.parR >> e) & 1ull)) return nullptr;
  OcrPlan* o = new OcrPlan();
  OcrArgs& a = o->a;
  o->mixed = mixed;
  o->DL = DL;
  o->nq = nq;
  a.D = (int)p.D;
  a.S = p.S;
  a.cols = cols;
  a.nbc = a.D / (DL * DL);
  a.K = t.K;
  a.sumd = t.sumd;
  a.sumdA = t.sumd + (t.sumd & 1);
  a.n1 = p.n1;
  a.np = (nq + 1) / 2;
  const bool pw2 = DL == 2 || DL == 4;
  auto pad = [&](long long x) { return (int)(pw2 ? x + (x >> 4) + (x >> 8) : x); };
  auto give_up = [&]() -> OcrPlan* { delete o; return nullptr; };
  // phases: pairs of modes, an odd last mode with its predecessor
  int pm[3][2];
  for (int q = 0; q < a.np; ++q) {
    pm[q][0] = std::min(2 * q, nq - 2);
    pm[q][1] = pm[q][0] + 1;
    OcrPhase& P = a.ph[q];
    P = OcrPhase{};
    P.mR = P.mL = P.expR = P.mR2 = P.mL2 = P.mE = P.expL = P.bA = P.bB = -1;
  }
  for (int i = 0; i < nq; ++i) a.eoff[i] = t.eoff[i];
  a.flip = t.flip;
  auto flip = [&](int mode) { return (int)((t.flip >> mode) & 1u); };
  auto matrix = [&](int mode, int op, int part, int J) {
    const int off = t.opd_off[mode] + op * DL * DL;
    for (int m = 0; m < a.nmat; ++m)
      if (a.m_off[m] == off && a.m_J[m] == J) return m;
    if (a.nmat == kRMat) return -1;
    a.m_off[a.nmat] = off;
    a.m_part[a.nmat] = part;
    a.m_flip[a.nmat] = flip(mode);
    a.m_J[a.nmat] = J;
    a.m_sign[a.nmat] = J >= 0 && (part ^ flip(mode)) ? -1 : 1;     // i A (x) i B = -A (x) B
    return a.nmat++;
  };
  auto phase_of = [&](int i, int j) {                // a phase that holds both modes, the last such
    for (int q = a.np - 1; q >= 0; --q)
      if ((pm[q][0] == i || pm[q][1] == i) && (pm[q][0] == j || pm[q][1] == j)) return q;
    return -1;
  };
  // couplings within a pair first (their right factor can be passed on too)
  for (int e = 0; e < p.ne; ++e) {
    const int q = phase_of(p.e_a[e], p.e_b[e]);
    if (q < 0) continue;
    const bool fwd = p.e_a[e] == pm[q][0];
    const int opl = fwd ? t.e_opa[e] : t.e_opb[e], opr = fwd ? t.e_opb[e] : t.e_opa[e];
    const int L = matrix(pm[q][0], opl, fwd ? t.e_pa[e] : t.e_pb[e], e);
    const int Rm = matrix(pm[q][1], opr, fwd ? t.e_pb[e] : t.e_pa[e], -1);
    OcrPhase& P = a.ph[q];
    if (L < 0 || Rm < 0) return give_up();
    if (P.mR < 0) { P.mR = Rm; P.mL = L; }
    else if (P.mR2 < 0) { P.mR2 = Rm; P.mL2 = L; }
    else return give_up();
  }
  // couplings between phases: the earlier phase writes the image w = B u of its mode, the
  // later one multiplies it by J A.  An image buffer is free again after its last reader
  // (which may be the phase that overwrites it: its threads read their own places first).
  struct Img { int phase, mat, last; bool right; };
  int held[kRBuf];                                    // last phase that reads buffer b, -1: free
  for (int& x : held) x = -1;
  for (int q = 0; q < a.np; ++q) {
    // images that phase q writes: (matrix on a or b) -> consumers
    struct Need { int mat; bool right; int last; std::vector<std::pair<int, std::pair<int, int>>> to; };
    std::vector<Need> need;
    for (int e = 0; e < p.ne; ++e) {
      if (phase_of(p.e_a[e], p.e_b[e]) >= 0) continue;
      // the phases of the two ends: the producer is the last phase that holds the earlier end
      int ph_a = -1, ph_b = -1;
      for (int r = 0; r < a.np; ++r) {
        if (pm[r][0] == p.e_a[e] || pm[r][1] == p.e_a[e]) { if (ph_a < 0) ph_a = r; }
        if (pm[r][0] == p.e_b[e] || pm[r][1] == p.e_b[e]) { if (ph_b < 0) ph_b = r; }
      }
      const bool a_first = ph_a < ph_b;
      const int src = a_first ? ph_a : ph_b, dst = a_first ? ph_b : ph_a;
      if (src == dst) return give_up();
      if (src != q) continue;
      const int ms = a_first ? p.e_a[e] : p.e_b[e], md = a_first ? p.e_b[e] : p.e_a[e];
      const int ops = a_first ? t.e_opa[e] : t.e_opb[e], opd = a_first ? t.e_opb[e] : t.e_opa[e];
      const int mat = matrix(ms, ops, a_first ? t.e_pa[e] : t.e_pb[e], -1);
      const int mJ = matrix(md, opd, a_first ? t.e_pb[e] : t.e_pa[e], e);
      if (mat < 0 || mJ < 0) return give_up();
      const bool right = ms == pm[q][1];
      Need* n = nullptr;
      for (Need& x : need) if (x.mat == mat && x.right == right) n = &x;
      if (!n) { need.push_back(Need{mat, right, dst, {}}); n = &need.back(); }
      n->last = std::max(n->last, dst);
      n->to.push_back({dst, {mJ, md == pm[dst][0] ? 1 : 0}});
    }
    OcrPhase& P = a.ph[q];
    for (Need& n : need) {
      int b = -1;
      for (int x = 0; x < kRBuf; ++x) if (held[x] <= q) { b = x; break; }
      if (b < 0) return give_up();
      held[b] = n.last;
      a.nbuf = std::max(a.nbuf, b + 1);
      if (n.right) {
        // the pair's own coupling computes R u already when the factors agree
        if (P.expR >= 0) return give_up();
        if (P.mR >= 0 && P.mR != n.mat) {
          if (P.mR2 == n.mat) { std::swap(P.mR, P.mR2); std::swap(P.mL, P.mL2); }
          else if (P.mR2 < 0) { P.mR2 = P.mR; P.mL2 = P.mL; P.mR = n.mat; P.mL = -1; }
          else return give_up();
        } else if (P.mR < 0) {
          P.mR = n.mat;
        }
        P.expR = b;
      } else {
        if (P.mE >= 0) return give_up();
        P.mE = n.mat;
        P.expL = b;
      }
      for (auto& to : n.to) {
        OcrPhase& T = a.ph[to.first];
        if (T.nimp == kRImp) return give_up();
        T.imp_buf[T.nimp] = b;
        T.imp_mat[T.nimp] = to.second.first;
        T.imp_a[T.nimp] = to.second.second;
        ++T.nimp;
      }
    }
  }
  // one-body slots, each in the first phase that holds its mode
  for (int u = 0; u < p.n1; ++u) {
    for (int q = 0; q < a.np; ++q) {
      OcrPhase& P = a.ph[q];
      if (pm[q][0] == p.s1_mode[u] && P.bA < 0) { P.bA = u; break; }
      if (pm[q][1] == p.s1_mode[u] && P.bB < 0) { P.bB = u; break; }
    }
    a.d_start[u] = t.drv_start[u];
    a.d_flip[u] = flip(p.s1_mode[u]);
    for (int x = t.drv_start[u]; x < t.drv_start[u + 1]; ++x) {
      a.d_drv[x] = t.drv_list[x];
      a.d_off[x] = t.opd_off[p.s1_mode[u]] + t.drv_op[t.drv_list[x]] * DL * DL;
    }
  }
  a.d_start[p.n1] = t.drv_start[p.n1];
  // One column per CTA, or as many as fill one warp: the columns are independent, so small
  // CTAs put a solve on more SMs and wait on fewer warps at every barrier.
  const int SC = std::max(1, 32 / a.nbc), NT = (SC * a.nbc + 31) / 32 * 32;      // Lay<DL, NQ>
  const int CS = (pad(a.D - 1) + 2) / 2 * 2;
  a.Sc = std::min(cols, SC);
  a.ncta = (cols + a.Sc - 1) / a.Sc;
  const int MS = DL * zrow(DL), nB = p.n1 * MS;
  if (NT > 256 || nB > kROne * NT) return give_up();
  const size_t cs = mixed ? sizeof(float2) : sizeof(double2), zs = 8;
  const size_t img = (size_t)SC * CS * cs, own = (size_t)DL * DL * NT * cs;
  size_t at = 0;
  auto take = [&](size_t b) { const size_t r = at; at = al16(at + b); return (int)r; };
  a.s_img = take(a.np > 1 ? (2 + a.nbuf) * img : 0);
  a.s_psi = take((size_t)DL * DL * NT * sizeof(double2));
  const bool reg = mixed && DL <= 4;
  a.s_b = take(reg ? 0 : own);
  a.s_acc = take(reg ? 0 : own);
  a.s_Q = take(reg ? 0 : own);
  a.s_mat = take((size_t)std::max(1, a.nmat) * MS * zs);
  a.s_one = take(2 * (size_t)std::max(1, nB) * zs);
  a.s_ph = take(2 * (size_t)a.sumdA * cs);
  o->smem = at;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (at + 1024 > (size_t)std::max(0, optin)) return give_up();
  // cross-density slots
  OcdArgs& g = o->dens;
  g.D = a.D; g.cols = cols; g.nbc = a.nbc; g.CS = CS; g.K = t.K; g.sumd = t.sumd; g.n1 = p.n1; g.ne = p.ne;
  bool fits = true;
  auto lay = [&](OcdSlot& S, int i, int j) {          // the slot's digit i, partner digit j
    S.s1 = pad(p.st[i]);
    S.s2 = pad(p.st[j]);
    std::vector<int> rest, ord;
    for (int k = nq - 1; k >= 0; --k) if (k != i && k != j) rest.push_back(k);
    for (int par = 0; par < 2; ++par)
      for (int k : rest) if ((nq - 1 - k) % 2 == par) { ord.push_back(k); break; }
    for (int k : rest) if (std::find(ord.begin(), ord.end(), k) == ord.end()) ord.push_back(k);
    S.no = (int)ord.size();
    for (int k = 0; k < S.no; ++k) S.pst[k] = pad(p.st[ord[k]]);
  };
  auto slot = [&]() -> OcdSlot* {
    if (g.nslot == kRSlot) { fits = false; return nullptr; }
    OcdSlot& S = g.slot[g.nslot++];
    S = OcdSlot{};
    S.sign = 1;
    S.mat = -1;
    return &S;
  };
  auto dmat = [&](int mode, int op, int part, int J) {
    if (g.nmat == kRMat) { fits = false; return 0; }
    g.m_off[g.nmat] = t.opd_off[mode] + op * DL * DL;
    g.m_part[g.nmat] = part;
    g.m_flip[g.nmat] = flip(mode);
    g.m_J[g.nmat] = J;
    g.m_sign[g.nmat] = part ^ flip(mode) ? -1 : 1;
    return g.nmat++;
  };
  for (int u = 0; u < p.n1 && fits; ++u)
    for (int x = t.drv_start[u]; x < t.drv_start[u + 1] && fits; ++x) {
      OcdSlot* S = slot();
      if (!S) break;
      const int i = p.s1_mode[u];
      S->drv = t.drv_list[x];
      S->mslot = u;
      S->off = t.opd_off[i] + t.drv_op[S->drv] * DL * DL;
      S->part = S->flip = flip(i);
      lay(*S, i, i ? i - 1 : 1);
    }
  const int ndrv = g.nslot;
  for (int e = 0; e < p.ne && fits; ++e)
    for (int side = 0; side < 2 && fits; ++side) {
      OcdSlot* S = slot();
      if (!S) break;
      const int i = side ? p.e_b[e] : p.e_a[e], j = side ? p.e_a[e] : p.e_b[e];
      S->kind = 1;
      S->edge = e;
      S->side = side;
      S->part = side ? t.e_pb[e] : t.e_pa[e];
      S->flip = flip(i);
      S->sign = S->part ^ S->flip ? -1 : 1;
      S->off = t.opd_off[i] + (side ? t.e_opb[e] : t.e_opa[e]) * DL * DL;
      S->mat = dmat(j, side ? t.e_opa[e] : t.e_opb[e], side ? t.e_pa[e] : t.e_pb[e], side ? e : -1);
      lay(*S, i, j);
    }
  if (fits) {
    g.Cg = std::max(1, std::min(cols, 4096 / a.D));
    g.ncg = (cols + g.Cg - 1) / g.Cg;
    const long long MD2 = SG_MAXD * SG_MAXD;
    g.accd = 2 * (long long)t.K * MD2 + 4 * (long long)p.ne * MD2 + (long long)p.n1 * SG_MAXD +
             2 * (long long)p.ne * SG_MAXD + p.ne;
    size_t q = 0;
    auto room = [&](size_t b) { const size_t r = q; q = al16(q + b); return (int)r; };
    // whole steps per load while they are small (the lanes then cover several images), else
    // one image at a time
    g.ni = g.Cg * a.nbc < 32 ? 4 * std::max(1, 512 / (4 * g.Cg * a.D)) : 1;
    g.s_img = room((size_t)2 * 2 * g.ni * g.Cg * g.CS * cs);
    g.s_mat = room((size_t)std::max(1, g.nmat) * MS * 8);
    g.s_g = room((size_t)kRSlot * 32 * 8);
    o->dsmem = q;
    o->dgrid = std::max(1, 304 / g.ncg);
    fits = q + 1024 <= (size_t)optin;
  }
  o->dens_ok = fits;
  o->ndrv = ndrv;
  o->half.D = a.D;
  o->half.nq = nq;
  o->half.DL = DL;
  for (int i = 0; i < nq; ++i) o->half.eoff[i] = t.eoff[i];
  return o;
}

void ocr_plan_destroy(OcrPlan* o) { delete o; }
int ocr_ctas(const OcrPlan* o) { return o->a.ncta; }

// Solves of equal signature share a launch, whose kernel reads the first one's arguments: all of them.
void ocr_signature(const OcrPlan* o, std::vector<long long>& sig) {
  static_assert(std::has_unique_object_representations_v<OcrArgs> && sizeof(OcrArgs) % sizeof(int) == 0);
  int v[sizeof(OcrArgs) / sizeof(int)];
  std::memcpy(v, &o->a, sizeof v);
  sig.insert(sig.end(), v, v + sizeof v / sizeof v[0]);
}

void ocr_half_step(const OcrPlan* o, const double* E, double dt, void* q, cudaStream_t st) {
  HalfArgs h = o->half;
  h.dt = dt;
  h.E = E;
  const int grid = (h.D + 63) / 64;
  if (o->mixed) k_ocr_half<float><<<grid, 64, 0, st>>>(h, (float2*)q);
  else k_ocr_half<double><<<grid, 64, 0, st>>>(h, (double2*)q);
}

namespace {
__global__ void k_ocr_many(OcrMany m, int nsys, int N, int K, int sumd, int D, int S, OcSys* __restrict__ t) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nsys; b += gridDim.x * blockDim.x) {
    OcSys d{};
    d.coef = m.coef + (size_t)b * 3 * N * K;
    d.ph = m.ph + (size_t)b * N * sumd;
    d.phmid = 1;
    d.half = m.half + (size_t)b * D;
    d.opd64 = m.opd + (size_t)b * m.opd_n;
    d.J = m.J + (size_t)b * m.J_n;
    d.psi_api = d.psi_out = m.psi + (size_t)b * D * S;
    d.K = 1;
    d.n1 = N;
    d.C = 1;
    d.L = N;
    t[b] = d;
  }
}
}  // namespace

size_t ocr_many_bytes(int nsys) { return (size_t)nsys * sizeof(OcSys); }

cudaError_t ocr_many(const OcrPlan* o, const OcrMany& m, int nsys, int N, double dt, void* table, cudaStream_t st) {
  k_ocr_many<<<(nsys + 63) / 64, 64, 0, st>>>(m, nsys, N, o->a.K, o->a.sumd, o->a.D, o->a.S, (OcSys*)table);
  OcBatch bt{};
  bt.nsys = nsys;
  bt.many = static_cast<const OcSys*>(table);
  bt.per = o->a.ncta;
  ocr_forward(o, bt, dt, st);
  return cudaGetLastError();
}

bool ocr_adjoint_ok(const OcrPlan* o) { return o->dens_ok; }
int ocr_blocks(const OcrPlan* o) { return o->dgrid * o->dens.ncg; }
int ocr_groups(const OcrPlan* o) { return o->dens.ncg; }


int ocr_densities(const OcrPlan* o, const void* u, const void* k, const void* coef, const double2* opd, const double* J,
                  int n0, int n1, double dt, bool ham, long long nstK, double* gF, double* acc, cudaStream_t st) {
  OcdArgs g = o->dens;
  g.ham = ham ? 1 : 0;
  g.nstK = nstK;
  if (!ham) g.nslot = o->ndrv;                         // the couplings' sides come last
  if (g.nslot == 0) return 0;
  const OcdJob j{u, k, coef, opd, J, gF, acc, n0, n1, dt};
  return o->mixed ? ocr_dens_f32(o, g, j, st) : ocr_dens_f64(o, g, j, st);
}

int ocr_forward(const OcrPlan* o, OcBatch& bt, double dt, cudaStream_t st) {
  return o->mixed ? ocr_fwd_f32(o, &bt, dt, st) : ocr_fwd_f64(o, &bt, dt, st);
}
int ocr_resident(const OcrPlan* o) {
  return o->mixed ? ocr_fwd_f32(o, nullptr, 0.0, nullptr) : ocr_fwd_f64(o, nullptr, 0.0, nullptr);
}

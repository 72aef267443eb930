// dg_fixed64_gl.cuh -- the FP64 element kernels on Gauss-Legendre nodes with
// their line sums, surface sums and face interpolations in 64-bit fixed point
// (see dg_fixed64.cuh for the numbers and why; the work is that of
// k_lift_gl and k_volume_gl in dg_stage_gl.cuh, which FP32-bulk uses).
// Measured per launch on 12^3 elements, N = 7 (0.88 M nodes): lifting
// 864 -> 336 us, volume kernel 549 -> 271 us; error against the long-double
// oracle 0.79 of the FP64 kernels' in the geometric mean, at most 0.999 in any
// variable (N = 1 .. 7, Ma 0.1 - 1.25).
#pragma once

namespace dg {

// The slot (face f, face point pq) a thread loads: side record and sign
template <int n>
__device__ __forceinline__ FaceRef slot_ref(const StageArgs& a, int e, int slot) {
  constexpr int n2 = n * n;
  return face_ref<n>(a, e, slot / n2, slot % n2 % n, slot % n2 / n);
}

// ---------------------------------------------------------------------------
// Lifted gradients and their ProlongToFace
// ---------------------------------------------------------------------------
// shared memory: Dhat's table, l / w and l at the ends, Dhat's table in FP64,
// the reduction words, then per element the planes of k_lift_fx (q and J planes: also the six
// faces' lifting fluxes [12][6 n2]; W planes: also the gradients)
template <int N>
struct LiftGlFix {
  using F = Fix<N>;
  static constexpr int ntab = LiftFix<N>::ntab + 4 * F::n;
  static constexpr int nqj = 10 * F::Pn > 72 * F::n2 ? 10 * F::Pn : 72 * F::n2;
  static constexpr int per_elem = nqj + 12 * F::Pn;
  static constexpr int Q = 20, nred = F::W * Q + 20 + 12 + 1;
  static constexpr size_t head(int epb) { return (8 * (ntab + LiftFix<N>::ntab) + 4 * (size_t)epb * nred + 15) & ~size_t(15); }
  static constexpr size_t bytes(int epb) { return head(epb) + 8 * (size_t)epb * per_elem; }
};

// the volume sums of a block with elements whose sums are taken in FP64;
// whether this element's are (out of line)
template <int N>
__device__ __noinline__ bool lift_gl_mixed(const Ops* o, const double* Me, long long* q, long long* J, long long* W, Fx* sD,
                                           double* sDd, unsigned* fin, unsigned* flag, bool bad, int t) {
  const int eq[4] = {fx_exp(fin[0]), fx_exp(fin[1]), fx_exp(fin[2]), fx_exp(fin[3])};
  const int eJ[3] = {fx_exp(fin[4]), fx_exp(fin[5]), fx_exp(fin[6])};
  const SumForm form = lift_form<N>(bad, q, fin, t, flag);
  if (!form.all) lift_sums_fx<N>(Me, q, J, W, sD, t, eq, eJ, form.direct);
  if (form.any)
    lift_sums_f64<N>(o, Me, reinterpret_cast<const double*>(q), reinterpret_cast<double*>(J),
                     reinterpret_cast<double*>(W), sDd, t, !form.direct);
  return form.direct;
}

template <int N>
__global__ void __launch_bounds__(Fix<N>::TPE * Fix<N>::D, Fix<N>::min_blocks(Fix<N>::TPE * Fix<N>::D))
    k_lift_gl_fx(StageArgs a) {
  using F = Fix<N>;
  using L = LiftGlFix<N>;
  constexpr int n = F::n, n2 = F::n2, n3 = F::n3, TPE = F::TPE, Pn = F::Pn;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / TPE, le = threadIdx.x / TPE, t = threadIdx.x % TPE;
  Fx* sD = reinterpret_cast<Fx*>(smraw);
  Fx* sL = sD + LiftFix<N>::ntab;  // [2][n] l(-1) / w, l(+1) / w
  Fx* sE = sL + 2 * n;             // [2][n] l(-1), l(+1)
  double* sDd = reinterpret_cast<double*>(sE + 2 * n);  // (filled by lift_sums_f64)
  unsigned* red = reinterpret_cast<unsigned*>(sDd + LiftFix<N>::ntab) + le * L::nred;
  unsigned* fin = red + F::W * L::Q;  // [20] maxima of the lifting
  unsigned* fing = fin + 20;          // [12] of the gradients
  unsigned* flag = fing + 12;
  long long* q = reinterpret_cast<long long*>(smraw + L::head(epb)) + (size_t)le * L::per_elem;
  long long* J = q + 4 * Pn;
  long long* Fl = q;           // [12][6 n2] the faces' lifting fluxes (after the volume sums)
  long long* W = q + L::nqj;   // [12][Pn]
  const ElemRef er = elem_ref(a, blockIdx.x * epb + le);
  const int e = er.e;
  const double* Me = a.metric + (size_t)e * 10 * n3;
  lift_table_fx<N>(a.ops, sD);
  for (int k = threadIdx.x; k < 2 * n; k += blockDim.x) sL[k] = fx_split(a.ops->fxL[k]), sE[k] = fx_split(a.ops->fxE[k]);
  prefetch_next64<N>(a, (blockIdx.x + a.prefetch) * epb + le, t - 32);
  if (t == 0) *flag = 0u;
  {
    unsigned m[20];  // those of lift_prims_fx, then the faces' fluxes, each of the 12 by itself
    lift_prims_fx<N>(a, e, q, m, t);
#pragma unroll
    for (int k = 8; k < 20; ++k) m[k] = 0;
    for (int s = t; s < 6 * n2; s += TPE) {
      const FaceRef r = slot_ref<n>(a, e, s);
      const double* Lr = a.lflux + (size_t)r.s * 12 * n2 + r.pqm;
#pragma unroll
      for (int k = 0; k < 12; ++k) m[8 + k] = max(m[8 + k], fx_mag(Lr[k * n2]));
    }
    fx_reduce<N, 20>(m, red, fin, t);
    __syncthreads();
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 20; ++k) bad = bad || (k != 7 && fx_bad(fin[k]));
  const int eq[4] = {fx_exp(fin[0]), fx_exp(fin[1]), fx_exp(fin[2]), fx_exp(fin[3])};
  const int eJ[3] = {fx_exp(fin[4]), fx_exp(fin[5]), fx_exp(fin[6])};
  if (lift_plain<N>(bad, fin)) lift_sums_fx<N>(Me, q, J, W, sD, t, eq, eJ, false);
  else bad = lift_gl_mixed<N>(a.ops, Me, q, J, W, sD, sDd, fin, flag, bad, t);
  // the six faces' lifting fluxes q* (s n), signed for this element (the
  // slave's outward normal is minus the master's), in its face frames
  for (int s = t; s < 6 * n2; s += TPE) {
    const FaceRef r = slot_ref<n>(a, e, s);
    const double* Lr = a.lflux + (size_t)r.s * 12 * n2 + r.pqm;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double x = r.slave ? -Lr[k * n2] : Lr[k * n2];
      Fl[k * 6 * n2 + s] = bad ? __double_as_longlong(x) : fx_from<60>(x, fx_exp(fin[8 + k]));
    }
  }
  __syncwarp();
  __syncthreads();
  unsigned mg[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) mg[k] = 0;
  for (int v = t; v < n3; v += TPE) {
    const int pv = fx_pad<n>(v);
    const int idx[3] = {v % n, (v / n) % n, v / n2};
    double acc[12];
    if (bad) {
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = __longlong_as_double(W[k * Pn + pv]);
      const double* Fd = reinterpret_cast<const double*>(Fl);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int pq = line_face_pq<n>(d, idx);
        const double cm = a.ops->Lm[idx[d]] * a.ops->winv[idx[d]], cp = a.ops->Lp[idx[d]] * a.ops->winv[idx[d]];
#pragma unroll
        for (int k = 0; k < 12; ++k)
          acc[k] += cm * Fd[k * 6 * n2 + 2 * d * n2 + pq] + cp * Fd[k * 6 * n2 + (2 * d + 1) * n2 + pq];
      }
    } else {
      // spread over the lines with l(+-1) / w: 6 2^(60 + 60 - 64 + 2) < 2^60.6
      Fx c[6];
      int at[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        c[f] = sL[(f & 1) * n + idx[f >> 1]];
        at[f] = f * n2 + line_face_pq<n>(f >> 1, idx);
      }
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        FxSum<2> s;
#pragma unroll
        for (int f = 0; f < 6; ++f) s.add(c[f], fx_split(Fl[k * 6 * n2 + at[f]]));
        const int pV = a.ops->fxH_bits - 2 - eq[k / 3] - eJ[k % 3];
        const int pS = a.ops->fxL_bits + 60 - 64 + 2 - fx_exp(fin[8 + k]);
        const int p = min(pV, pS);
        acc[k] = fx_to(fx_shr(W[k * Pn + pv], min(pV - p, 62)) + fx_shr(s.get(), min(pS - p, 62)), p);
      }
    }
    const double Ji = Me[9 * n3 + v];
    double* g = a.g + (size_t)e * 12 * n3 + v;
    double* Wd = reinterpret_cast<double*>(W) + pv;  // (this thread's own nodes)
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      acc[k] *= Ji;
      if (er.valid) g[k * n3] = acc[k];
      Wd[k * Pn] = acc[k];
      mg[k] = max(mg[k], fx_mag(acc[k]));
    }
  }
  fx_reduce<N, 12>(mg, red, fing, t);
  __syncthreads();
  bool gbad = false;
#pragma unroll
  for (int k = 0; k < 12; ++k) gbad = gbad || fx_bad(fing[k]);
  if (!gbad)
    for (int v = t; v < n3; v += TPE) {
      long long* x = W + fx_pad<n>(v);
#pragma unroll
      for (int k = 0; k < 12; ++k) x[k * Pn] = fx_from<60>(__longlong_as_double(x[k * Pn]), fx_exp(fing[k]));
    }
  __syncwarp();
  __syncthreads();
  if (!er.valid) return;
  // ProlongToFace of the gradients
  for (int s = t; s < 6 * n2; s += TPE) {
    const int f = s / n2;
    int v0, st;
    face_line<n>(f, s % n2 % n, s % n2 / n, v0, st);
    const FaceRef r = slot_ref<n>(a, e, s);
    double* o = a.gfc + ((size_t)r.s * 2 + (r.slave ? 1 : 0)) * 12 * n2 + r.pqm;
    if (gbad) {
      const double* Lv = (f & 1) ? a.ops->Lp : a.ops->Lm;
      const double* Wd = reinterpret_cast<const double*>(W);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        double val = 0.0;
        for (int al = 0; al < n; ++al) val += Lv[al] * Wd[k * Pn + fx_pad<n>(v0 + al * st)];
        o[k * n2] = val;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        FxSum<3> x;  // 2^(62 + 60 - 64 + 3)
#pragma unroll
        for (int al = 0; al < n; ++al) x.add(sE[(f & 1) * n + al], fx_split(W[k * Pn + fx_pad<n>(v0 + al * st)]));
        o[k * n2] = fx_to(x.get(), a.ops->fxE_bits + 60 - 64 + 3 - fx_exp(fing[k]));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Volume integral (collocated flux divergence) + SurfInt + ApplyJac (+ RK)
// ---------------------------------------------------------------------------
// A node's fluxes are a tensor T (rho u; rho u u + p - tau, symmetric; rho u H
// - W: 12 numbers in FP64), contracted with each direction's metrics.  The
// metrics have an exponent eJ for each Cartesian component (over the three
// directions), each of T's five rows one exponent for its three values scaled
// by 2^(eJ_j), so that the products of a row meet in one scale whatever the
// element's stretching (15 numbers).
// shared memory: Dhat, l / w at the ends, the reduction words, then per
// element the fluxes of one direction (5 planes), the tensor (15 planes) and
// the six faces' surface fluxes [5][6 n2]
// the place of row r, column j among the 12 numbers
__device__ __forceinline__ constexpr int gl_at(int r, int j) {
  return r == 0 ? j : r == 4 ? 9 + j : r - 1 == j ? 3 + j : 4 + r + j;  // xx, yy, zz, xy, xz, yz from 3 on
}

template <int N>
struct VolGlFix {
  using F = Fix<N>;
  static constexpr int ntab = F::n2 + 2 * F::n;
  static constexpr int offT = 5 * F::Pn, offS = offT + 15 * F::n3, per_elem = offS + 30 * F::n2;
  // maxima: T; metrics by component; the five f*; density, pressure and rho H and their complements (minima); flag
  static constexpr int Q = 26, nred = F::W * Q + Q + 1;
  static constexpr size_t head(int epb) { return (8 * ntab + 4 * (size_t)epb * nred + 15) & ~size_t(15); }
  static constexpr size_t bytes(int epb) { return head(epb) + 8 * (size_t)epb * per_elem; }
};

// whether the element's sums are taken in FP64 (as vol_form; out of line)
template <int N>
__device__ __noinline__ bool vol_gl_direct(const double* u, double gm1, const unsigned* fin, bool bad, int t, unsigned* flag) {
  constexpr int n = Fix<N>::n, n3 = Fix<N>::n3;
  const unsigned cR = fx_cut(fin[20]), cP = fx_cut(fin[21]), cH = fx_cut(fin[22]);
  auto level = [=](int v, int k) {
    double U[5];
    for (int i = 0; i < 5; ++i) U[i] = u[i * n3 + v];
    const double p = prim64(U, gm1).p;
    return fx_mag(k == 0 ? U[0] : k == 1 ? p : U[4] + p);
  };
  auto rho = [=](int v) { return level(v, 0); };
  auto prs = [=](int v) { return level(v, 1); };
  auto rhoH = [=](int v) { return level(v, 2); };
  return sum_form<N>(bad, t, flag, [=](int v) {
           return (rho(v) < cR && lines_quiet<n>(v, cR, rho)) || (prs(v) < cP && lines_quiet<n>(v, cP, prs)) ||
                  (rhoH(v) < cH && lines_quiet<n>(v, cH, rhoH));
         }).direct;
}

template <int N, int MODE>
__global__ void __launch_bounds__(Fix<N>::TPE * Fix<N>::D, Fix<N>::min_blocks(Fix<N>::TPE * Fix<N>::D))
    k_volume_gl_fx(StageArgs a) {
  using F = Fix<N>;
  using L = VolGlFix<N>;
  constexpr int n = F::n, n2 = F::n2, n3 = F::n3, TPE = F::TPE, Pn = F::Pn, R = F::R;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / TPE, le = threadIdx.x / TPE, t = threadIdx.x % TPE;
  Fx* sDh = reinterpret_cast<Fx*>(smraw);
  Fx* sL = sDh + n2;
  unsigned* red = reinterpret_cast<unsigned*>(sL + 2 * n) + le * L::nred;
  unsigned* fin = red + F::W * L::Q;
  unsigned* flag = fin + L::Q;
  long long* G = reinterpret_cast<long long*>(smraw + L::head(epb)) + (size_t)le * L::per_elem;  // [5][Pn]
  long long* T = G + L::offT;   // [15][n3] (in FP64 the first 12)
  long long* Fs = G + L::offS;  // [5][6 n2]
  const ElemRef er = elem_ref(a, blockIdx.x * epb + le);
  const int e = er.e;
  const CaseParams cp = case_params(a, 0);
  const double* Me = a.metric + (size_t)e * 10 * n3;
  for (int k = threadIdx.x; k < n2; k += blockDim.x) {
    sDh[k] = fx_split(a.ops->fxH[k]);
    if (k < 2 * n) sL[k] = fx_split(a.ops->fxL[k]);
  }
  if (t == 7 && MODE == 1 && !a.first_stage) prefetch64(a.dU, (size_t)e * 5 * n3, 5 * n3);
  prefetch_next64<N>(a, (blockIdx.x + a.prefetch) * epb + le, t - 32);
  if (t == 0) *flag = 0u;
  {
    unsigned m[L::Q];
#pragma unroll
    for (int k = 0; k < L::Q; ++k) m[k] = 0;
    for (int v = t; v < n3; v += TPE) {
      double U[5], tau[6] = {0, 0, 0, 0, 0, 0}, W[3] = {0, 0, 0};
      load_state64<n>(a, e, v, U);
      const Prim64 pr = prim64(U, a.gm1);
      if (a.viscous) {
        double g[12], vmu, vlam;
        const double* pg = a.g + (size_t)e * 12 * n3 + v;
#pragma unroll
        for (int k = 0; k < 12; ++k) g[k] = pg[k * n3];
        visc_coeffs<double>(a, cp, a.sutherland ? pr.p * pr.ri * a.Rinv : 0.0, vmu, vlam);
        viscous_parts(g, pr.u, pr.v, pr.w, vmu, vlam, tau, W);
      }
      const double rH = U[4] + pr.p;
      double x[12];
      x[0] = U[1], x[1] = U[2], x[2] = U[3];
      x[3] = (U[1] * pr.u - tau[0]) + pr.p;  // xx, yy, zz, xy, xz, yz
      x[4] = (U[2] * pr.v - tau[1]) + pr.p;
      x[5] = (U[3] * pr.w - tau[2]) + pr.p;
      x[6] = U[1] * pr.v - tau[3], x[7] = U[1] * pr.w - tau[4], x[8] = U[2] * pr.w - tau[5];
      x[9] = rH * pr.u - W[0], x[10] = rH * pr.v - W[1], x[11] = rH * pr.w - W[2];
      double* Td = reinterpret_cast<double*>(T) + v;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        Td[k * n3] = x[k];
        m[k] = max(m[k], fx_mag(x[k]));
      }
      const unsigned lev[3] = {fx_mag(U[0]), fx_mag(pr.p), fx_mag(rH)};
#pragma unroll
      for (int k = 0; k < 3; ++k) m[20 + k] = max(m[20 + k], lev[k]), m[23 + k] = max(m[23 + k], ~lev[k]);
#pragma unroll
      for (int c = 0; c < 9; ++c) m[12 + c % 3] = max(m[12 + c % 3], fx_mag(Me[c * n3 + v]));
    }
    for (int s = t; s < 6 * n2; s += TPE) {
      const FaceRef r = slot_ref<n>(a, e, s);
      const double* src = a.fstar + (size_t)r.s * 5 * n2 + r.pqm;
#pragma unroll
      for (int k = 0; k < 5; ++k) m[15 + k] = max(m[15 + k], fx_mag(src[k * n2]));
    }
    fx_reduce<N, L::Q>(m, red, fin, t);
    __syncthreads();
  }
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 20; ++k) bad = bad || fx_bad(fin[k]);
  const int eJ[3] = {fx_exp(fin[12]), fx_exp(fin[13]), fx_exp(fin[14])};
  int eR[5];  // the rows' exponents
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    eR[r] = -4000;
#pragma unroll
    for (int j = 0; j < 3; ++j) eR[r] = max(eR[r], fx_exp(fin[gl_at(r, j)]) + eJ[j]);
  }
  {
    // FP64 sums where density, pressure or rho H are quiet on a node's lines (vol_form)
    bool ask = bad;
#pragma unroll
    for (int k = 0; k < 3; ++k) ask = ask || ~fin[23 + k] < fx_cut(fin[20 + k]);
    __syncwarp();
    if (blockDim.x == TPE ? ask : __syncthreads_or(ask)) bad = vol_gl_direct<N>(a.U + (size_t)e * 5 * n3, a.gm1, fin, bad, t, flag);
  }
  if (!bad)
    for (int v = t; v < n3; v += TPE) {
      double x[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) x[k] = __longlong_as_double(T[k * n3 + v]);
#pragma unroll
      for (int k = 0; k < 15; ++k) T[k * n3 + v] = fx_from<60>(x[gl_at(k / 3, k % 3)], eR[k / 3] - eJ[k % 3]);
    }
  // the six faces' fluxes f* s, signed for this element
  for (int s = t; s < 6 * n2; s += TPE) {
    const FaceRef r = slot_ref<n>(a, e, s);
    const double* src = a.fstar + (size_t)r.s * 5 * n2 + r.pqm;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double x = r.slave ? -src[k * n2] : src[k * n2];
      Fs[k * 6 * n2 + s] = bad ? __double_as_longlong(x) : fx_from<60>(x, fx_exp(fin[15 + k]));
    }
  }
  long long acc[R][5];
  double sum[R][5];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int k = 0; k < 5; ++k) acc[r][k] = 0, sum[r][k] = 0.0;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    for (int v = t; v < n3; v += TPE) {
      const int pv = fx_pad<n>(v);
      const double nv[3] = {Me[3 * d * n3 + v], Me[(3 * d + 1) * n3 + v], Me[(3 * d + 2) * n3 + v]};
      if (bad) {
        const double* Td = reinterpret_cast<const double*>(T) + v;
        double* Gd = reinterpret_cast<double*>(G) + pv;
        Gd[0] = Td[0] * nv[0] + Td[n3] * nv[1] + Td[2 * n3] * nv[2];
        Gd[Pn] = Td[3 * n3] * nv[0] + Td[6 * n3] * nv[1] + Td[7 * n3] * nv[2];
        Gd[2 * Pn] = Td[6 * n3] * nv[0] + Td[4 * n3] * nv[1] + Td[8 * n3] * nv[2];
        Gd[3 * Pn] = Td[7 * n3] * nv[0] + Td[8 * n3] * nv[1] + Td[5 * n3] * nv[2];
        Gd[4 * Pn] = Td[9 * n3] * nv[0] + Td[10 * n3] * nv[1] + Td[11 * n3] * nv[2];
      } else {
        const Fx j0 = fx_split(fx_from<60>(nv[0], eJ[0])), j1 = fx_split(fx_from<60>(nv[1], eJ[1])),
                 j2 = fx_split(fx_from<60>(nv[2], eJ[2]));
#pragma unroll
        for (int r = 0; r < 5; ++r) {
          const long long* x = T + 3 * r * n3 + v;
          FxSum<2> s;  // 3 2^(60 + 60 - 64 + 2) < 2^59.6
          s.add(fx_split(x[0]), j0), s.add(fx_split(x[n3]), j1), s.add(fx_split(x[2 * n3]), j2);
          G[r * Pn + pv] = s.get();
        }
      }
    }
    __syncwarp();
    __syncthreads();
    const int sd = dir_stride<n>(d);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int v = t + r * TPE;
      if (v < n3) {
        const int id = dir_index<n>(v, d), base = v - id * sd;
        if (bad) {
          const double* Gd = reinterpret_cast<const double*>(G);
          for (int al = 0; al < n; ++al)
#pragma unroll
            for (int k = 0; k < 5; ++k) sum[r][k] += a.ops->Dhat[id * n + al] * Gd[k * Pn + fx_pad<n>(base + al * sd)];
        } else {
          FxSum<3> s[5];  // 2^(62 + 59.6 - 64 + 3) per direction
#pragma unroll
          for (int al = 0; al < n; ++al) {
            const int pa = fx_pad<n>(base + al * sd);
            const Fx c = sDh[id * n + al];
#pragma unroll
            for (int k = 0; k < 5; ++k) s[k].add(c, fx_split(G[k * Pn + pa]));
          }
#pragma unroll
          for (int k = 0; k < 5; ++k) acc[r][k] += s[k].get();
        }
      }
    }
    __syncwarp();
    __syncthreads();
  }
  if (!er.valid) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int v = t + r * TPE;
    if (v >= n3) break;
    const int idx[3] = {v % n, (v / n) % n, v / n2};
    // SurfInt: the faces' fluxes spread over the lines with l(+-1) / w
    if (bad) {
      const double* Fd = reinterpret_cast<const double*>(Fs);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int pq = line_face_pq<n>(d, idx);
        const double cm = a.ops->Lm[idx[d]] * a.ops->winv[idx[d]], cpl = a.ops->Lp[idx[d]] * a.ops->winv[idx[d]];
#pragma unroll
        for (int k = 0; k < 5; ++k)
          sum[r][k] += cm * Fd[k * 6 * n2 + 2 * d * n2 + pq] + cpl * Fd[k * 6 * n2 + (2 * d + 1) * n2 + pq];
      }
    } else {
      Fx c[6];
      int at[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        c[f] = sL[(f & 1) * n + idx[f >> 1]];
        at[f] = f * n2 + line_face_pq<n>(f >> 1, idx);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        FxSum<2> s;  // 6 2^(60 + 60 - 64 + 2) < 2^60.6
#pragma unroll
        for (int f = 0; f < 6; ++f) s.add(c[f], fx_split(Fs[k * 6 * n2 + at[f]]));
        const int pV = a.ops->fxH_bits - 3 - eR[k];
        const int pS = a.ops->fxL_bits + 60 - 64 + 2 - fx_exp(fin[15 + k]);
        const int p = min(pV, pS);
        sum[r][k] = fx_to(fx_shr(acc[r][k], min(pV - p, 62)) + fx_shr(s.get(), min(pS - p, 62)), p);
      }
    }
    finish_node64<n, MODE, true>(a, e, er.ce, v, sum[r]);
  }
}

}  // namespace dg

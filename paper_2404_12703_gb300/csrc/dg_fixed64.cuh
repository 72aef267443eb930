// dg_fixed64.cuh -- the FP64 element kernels on LGL nodes with their line sums
// and two-point fluxes in 64-bit fixed point on the integer pipe (included by
// dg_stage.cuh).
//
// Why.  A GB300 SM finishes 1.96 FP64 operations per clock and 61 products
// 32 x 32 -> 64 bits with a 64-bit addition (mad.wide), 59 additions of 64-bit
// integers (measured).  A product of two 62-bit fixed-point numbers, rounded
// to 64 bits, is three mad.wide and a shift: eight times cheaper than one
// FP64 multiplication.  The kernels here were bound by the FP64 unit (84 - 96 %
// busy); what they keep on it is ConsToPrim, the stress tensor and the
// Runge-Kutta update.  Measured per launch on 24^3 elements, N = 7 (7.08 M
// nodes): volume kernel 7.70 -> 2.55 ms, lifting 4.12 -> 1.40 ms; now bound by
// latency at two blocks per SM.
//
// Numbers.  Every element scales each group of quantities (density, velocity,
// pressure, enthalpy, metrics by Cartesian component, ...) by the power of two
// that brings the group's largest magnitude in the element below 2^60 or 2^61;
// a value is that many bits of a two's complement 64-bit integer.  A conversion
// is off by less than one unit: 2^-59 of the group's largest value (2^-60 of
// density, pressure, enthalpy and the lifted variables, 2^-57 of the heat flux
// beside a large work term), where FP64 rounds each value to 2^-53 of itself.
// Products keep 64 bits, sums are exact, results are rounded to FP64 once.
// The largest values of a group so have more bits than FP64 gives them and
// those below a sixty-fourth fewer.  What that may cost, and what is done:
// - Different velocity components, metrics and stresses: groups or scalings by
//   component (lifting, vol_scale, the rows of dg_fixed64_gl.cuh), so that a
//   small cross-flow or a stretched element keeps its bits.
// - Density, pressure, energy or temperature that span more than a factor of
//   16 in an element: FP64 rounds a node's sums at the size of the largest
//   values on the node's three lines.  Where they miss the element's large
//   values (lines_quiet), the element is done in FP64.
// - Light and fast or hot fluid beside dense fluid, small components beside
//   hypersonic flow (vol_bad), stresses above the pressure: in FP64 too.
// - A non-finite value, or a group whose largest value is outside 2^-200 ..
//   2^200: in FP64, with its own treatment of such values.
// FP64 sums cost what they did before: a step whose elements all take them
// (density ratios of 1e6) has 0.78, 0.88, 0.87, 0.89, 0.97, 1.07 and 1.01 of the
// time it had in FP64 kernels, N = 1 .. 7; one without any 0.42 - 0.65.
// Scales depend on the element alone, so results do not depend on the launch
// shape.  The bounds on every intermediate value stand beside it; none can
// overflow.  Error of the right-hand side against the long-double oracle over
// that of the FP64 kernels, N = 1 .. 7, Ma 0.1 - 1.25, viscous, Roe and LF: 0.53
// in the geometric mean, at most 0.999 in any variable (Gauss nodes 0.79, 0.999).
#pragma once

namespace dg {

// A 64-bit integer x as hi 2^32 + lo with lo in [-2^31, 2^31)
struct Fx {
  int lo, hi;
};
__device__ __forceinline__ Fx fx_split(long long x) {
  const int lo = (int)x;
  return {lo, (int)(x >> 32) + (int)((unsigned)lo >> 31)};
}
// Sum of products a b 2^-64: h in units of 1, x in units of 2^-32 (the
// products of the low words, below half a unit each, are left out).  get: the
// sum times 2^S.  FxSum<S> rounds (x starts at half a unit of the result);
// FxSumS takes S at run time and truncates (the two nodes of a pair take the
// same truncated flux, so that nothing is gained or lost).
__device__ __forceinline__ long long fx_get(long long h, long long x, int S) {
  return (long long)((unsigned long long)h << S) + (x >> (32 - S));
}
template <int S>
struct FxSum {
  long long h = 0, x = 1LL << (31 - S);
  __device__ __forceinline__ void add(Fx a, Fx b) {
    h += (long long)a.hi * b.hi;
    x += (long long)a.hi * b.lo;
    x += (long long)a.lo * b.hi;
  }
  __device__ __forceinline__ long long get() const { return fx_get(h, x, S); }
};
struct FxSumS {
  long long h = 0, x = 0;
  __device__ __forceinline__ void add(Fx a, Fx b) {
    h += (long long)a.hi * b.hi;
    x += (long long)a.hi * b.lo;
    x += (long long)a.lo * b.hi;
  }
  __device__ __forceinline__ long long get(int S) const { return fx_get(h, x, S); }
};
// v 2^-k, rounded (k = 0 .. 62, |v| below 2^62)
__device__ __forceinline__ long long fx_shr(long long v, int k) { return (v + (long long)((1ull << k) >> 1)) >> k; }

// Biased FP64 exponent of the largest magnitude from the maximum of the high words
__device__ __forceinline__ unsigned fx_field(unsigned hi_max) { return hi_max >> 20; }
__device__ __forceinline__ unsigned fx_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
// exponents outside 2^-200 .. 2^200 (zero is inside)
__device__ __forceinline__ bool fx_bad(unsigned hi_max) {
  const unsigned f = fx_field(hi_max);
  return f > 1223u || (f < 823u && hi_max != 0u);
}
// e with every |v| of the group < 2^e (an all-zero group: the smallest)
__device__ __forceinline__ int fx_exp(unsigned hi_max) { return max((int)fx_field(hi_max), 823) - 1022; }

// v 2^(BITS - e), |v| < 2^e, truncated towards zero
template <int BITS>
__device__ __forceinline__ long long fx_from(double v, int e) {
  const int hi = __double2hiint(v);
  const int r = min(e + 1022 - ((hi >> 20) & 0x7ff), 63);  // >= 0 within the group
  const unsigned long long m =
      ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v)) << (BITS - 53);
  const long long q = (long long)(m >> (r & 63));
  const long long s = hi >> 31;
  return (q ^ s) - s;
}
// x 2^-p rounded to FP64 (|p| < 900)
__device__ __forceinline__ double fx_to(long long x, int p) {
  const long long s = x >> 63;
  const unsigned long long m = (unsigned long long)((x ^ s) - s);
  const int lz = __clzll((long long)m);
  const unsigned long long f = m << (lz & 63);                     // leading one at bit 63
  const unsigned long long q = (f >> 11) + ((f >> 10) & 1ull);     // 53 bits, rounded (a carry gives 2^53)
  // the implicit bit adds one to the exponent field
  const unsigned long long b = q + ((unsigned long long)(unsigned)(1023 + 63 - lz - p - 1) << 52);
  return m ? __longlong_as_double((long long)(b | ((unsigned long long)s & 0x8000000000000000ull))) : 0.0;
}

// a node plane with pads (fx_pad), an even number of words: planes of 16-byte
// pairs start 16-byte aligned behind any number of planes
template <int n>
__host__ __device__ constexpr int fx_plane() {
  return (n * n * n + n * n + n + 1) & ~1;
}

// Threads per element: a multiple of a warp (so that a warp's maxima are one
// element's) or, at N = 1, eight.  The two-point sums give each warp whole
// lines (LW lanes): the threads per element are those that leave few lanes
// idle there and in the node loops.
template <int N>
struct Fix {
  static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  static constexpr int TPE = n == 2 ? 8 : n == 3 ? 32 : n == 4 ? 64 : n == 5 ? 160 : n == 6 ? 128 : n == 7 ? 224 : 256;
  static constexpr int W = TPE >= 32 ? TPE / 32 : 1;            // warps per element
  static constexpr int LW = TPE >= 32 ? 32 / n * n : TPE;       // lanes of a warp (or element) that hold whole lines
  static constexpr int R = (n3 + TPE - 1) / TPE;                // nodes per thread
  static constexpr int RL = (n3 + W * LW - 1) / (W * LW);       // the same in whole lines per warp
  static constexpr int Pn = fx_plane<n>();
  static constexpr int D = Shape<N>::EPB_DEFAULT;
  static constexpr bool lift2 = 2 * D * n3 <= 1024, vol2 = 2 * D * n3 <= 512;
  // launch bounds: the largest block of the variants
  static constexpr int TL = TPE * (lift2 ? 2 * D : D), TV = TPE * (vol2 ? 2 * D : D);
  static constexpr int min_blocks(int threads) { return threads <= 256 ? 2 : 1; }
};

// padded plane index: one pad after each line and each layer of nodes, so
// that lines along all three directions fall in distinct banks
template <int n>
__device__ __forceinline__ int fx_pad(int v) {
  return v + v / n + v / (n * n);
}

// The maxima of Q values over the element's threads: each thread gives its
// own in m; they are in out[Q] (the element's shared memory) for the threads
// of the element's first warp when the call returns.  red: [W][Q] words.
template <int N, int Q>
__device__ __forceinline__ void fx_reduce(unsigned m[Q], unsigned* red, unsigned* out, int t) {
  using F = Fix<N>;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    if constexpr (F::TPE < 32) {
#pragma unroll
      for (int o = F::TPE / 2; o > 0; o >>= 1) m[k] = max(m[k], __shfl_xor_sync(0xffffffffu, m[k], o));
    } else {
      m[k] = __reduce_max_sync(0xffffffffu, m[k]);
    }
  }
  if (t % 32 == 0) {
#pragma unroll
    for (int k = 0; k < Q; ++k) red[(t / 32) * Q + k] = m[k];
  }
  __syncwarp();
  __syncthreads();
  if (t < 32)
    for (int k = t; k < Q; k += F::TPE < 32 ? F::TPE : 32) {
      unsigned x = red[k];
#pragma unroll
      for (int w = 1; w < F::W; ++w) x = max(x, red[w * Q + k]);
      out[k] = x;
    }
  __syncwarp();
}
// the largest magnitude of a group (its high word) over 2^e, from above
__device__ __forceinline__ float fx_frac(unsigned hi, int e) {
  const int x = (int)fx_field(hi) - 1022 - e;
  return hi == 0u || x < -100 ? 0.0f : __uint_as_float(((unsigned)(126 + x) << 23) | ((hi & 0xfffffu) << 3)) * 1.00001f;
}
// b 2^k, b >= 0, from above (k clamped to +-126)
__device__ __forceinline__ float fx_scale(float b, int k) { return b * __uint_as_float((unsigned)(127 + max(-126, min(126, k))) << 23); }
// the largest S in 0 .. 31 with b 2^S <= 2^top
__device__ __forceinline__ int fx_room(float b, int top) {
  const int l = (int)((__float_as_uint(b) + 0x7fffffu) >> 23) - 127;  // b <= 2^l
  return max(0, min(31, top - l));
}

// A magnitude's high word scaled by 2^-k (zero where it vanishes), the cut
// below which a value of a group is quiet (a sixteenth of the largest), and
// whether a node's three lines hold quiet values only.  Fixed point keeps a
// quiet value's bits below FP64's; where a line through the node holds a
// larger value, FP64 rounds the node's sums at that value's size anyway.
__device__ __forceinline__ unsigned fx_down(unsigned mag, int k) {
  return mag > (unsigned)k << 20 ? mag - ((unsigned)k << 20) : 0u;
}
__device__ __forceinline__ unsigned fx_cut(unsigned hi_max) { return fx_down(hi_max, 4); }
template <int n, class Mag>
__device__ __forceinline__ bool lines_quiet(int v, unsigned cut, Mag mag) {
  for (int d = 0; d < 3; ++d) {
    const int sd = dir_stride<n>(d), base = v - dir_index<n>(v, d) * sd;
    for (int al = 0; al < n; ++al)
      if (mag(base + al * sd) >= cut) return false;
  }
  return true;
}
// Which sums an element and its block take: direct (FP64), and whether any or
// all elements of the block do.  Blocks of plain elements run code of their own
// from here on, the others a copy out of line: beside each other in one body
// the FP64 form's registers cost the fixed-point one 1 to 8 % (volume kernel,
// 24^3, N = 7: 2,575 against 2,552 us; 16^3, N = 5: 373 against 345).
struct SumForm {
  bool direct, any, all;
};
// For a block that holds an element whose sums are taken in FP64 in any case
// (bad) or that has a node with a quiet value (the groups' minima tell).
// quiet(v): whether node v is quiet in a group on all its lines; flag: a word
// of the element's shared memory, zero when called.
template <int N, class Quiet>
__device__ __forceinline__ SumForm sum_form(bool bad, int t, unsigned* flag, Quiet quiet) {
  constexpr int n3 = Fix<N>::n3, TPE = Fix<N>::TPE;
  bool is = false;
  if (!bad)
    for (int v = t; v < n3; v += TPE) is = is || quiet(v);
  if (is) *flag = 1u;
  __syncwarp();
  __syncthreads();
  const bool direct = bad || *flag != 0u;
  __syncwarp();
  const bool any = __syncthreads_or(direct), all = __syncthreads_and(direct);
  return {direct, any, all};
}

template <int n>
__device__ __forceinline__ void load_state64(const StageArgs& a, int e, int v, double U[5]) {
  constexpr int n3 = n * n * n;
  const double* u = a.U + (size_t)e * 5 * n3 + v;
#pragma unroll
  for (int k = 0; k < 5; ++k) U[k] = u[k * n3];
}
template <int n>
__device__ __forceinline__ int line_base(int d, int l) {
  const int lp = l % n, lq = l / n;
  return d == 0 ? n * l : (d == 1 ? lp + n * n * lq : l);
}

// the element of a block's slot and whether its results are stored (slots
// past the end redo the last element; free slots of a serving pool and
// elements of cases that sit the step out store nothing)
struct ElemRef {
  int e, ce;
  bool valid, busy;
};
__device__ __forceinline__ ElemRef elem_ref(const StageArgs& a, int slot) {
  ElemRef r;
  const int ei = slot < a.E ? slot : a.E - 1;
  r.e = a.elem_list ? a.elem_list[ei] : ei;
  r.ce = a.elem_case ? a.elem_case[r.e] : 0;
  r.valid = slot < a.E && r.ce >= 0;
  r.busy = r.valid && !(a.cases && a.cases[r.ce].dt == 0.0);
  return r;
}

// Asks L2 for what an element block reads later on (its lifting fluxes or its
// gradients, register and surface fluxes), and for the state and metrics of
// the element a wave of blocks further on: each phase of a block then waits
// on L2 instead of on memory.  One thread per side or array.
template <int N>
__device__ __forceinline__ void prefetch_sides64(const StageArgs& a, int e, const double* base, int comps, int t) {
  constexpr int n2 = Fix<N>::n2;
  if (t < 6) {
    const size_t w = (size_t)comps * n2, s = (size_t)es_side(a.elem_side[(size_t)e * 6 + t]) * w;
    prefetch_l2(base + s, 8 * w, base + s, base + s + w);
  }
}
__device__ __forceinline__ void prefetch64(const double* base, size_t first, size_t count) {
  prefetch_l2(base + first, 8 * count, base + first, base + first + count);
}
template <int N>
__device__ __forceinline__ void prefetch_next64(const StageArgs& a, int slot, int t) {
  constexpr int n3 = Fix<N>::n3;
  if (slot < a.E && t >= 0 && t < 2) {
    const size_t e = a.elem_list ? a.elem_list[slot] : slot;
    if (t == 0) prefetch64(a.U, e * 5 * n3, 5 * n3);
    else prefetch64(a.metric, e * 10 * n3, 10 * n3);
  }
}

// ApplyJac of a node's sums s, the sources, and Ut or the RK update
template <int n, int MODE, bool EXTRA>
__device__ __forceinline__ void finish_node64(const StageArgs& a, int e, int ce, int v, const double s[5]) {
  constexpr int n3 = n * n * n;
  const double Ji = -a.metric[((size_t)e * 10 + 9) * n3 + v];
  double Ut[5], U[5];
  load_state64<n>(a, e, v, U);
  if constexpr (!EXTRA && MODE == 1) {  // (no sources: dt / J in one factor)
    const double c = Ji * case_dt(a, ce);
    double* du = a.dU + (size_t)e * 5 * n3 + v;
    double* uo = a.Urk + (size_t)e * 5 * n3 + v;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double x = a.first_stage ? s[k] * c : a.rkA * du[k * n3] + s[k] * c;
      du[k * n3] = x;
      uo[k * n3] = U[k] + a.rkB * x;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) Ut[k] = s[k] * Ji;
  if (EXTRA && a.sponge_sigma) {  // sponge source -sigma (U - U_base)
    const double sg = a.sponge_sigma[(size_t)e * n3 + v];
    const double* ub = a.sponge_base + (size_t)e * 5 * n3 + v;
#pragma unroll
    for (int k = 0; k < 5; ++k) Ut[k] -= sg * (U[k] - ub[k * n3]);
  }
  if (EXTRA && a.source) {  // manufactured-solution source
    double Q[5];
    mms_source(a, a.xyzs + ((size_t)e * n3 + v) * 3, stage_time(a, MODE), Q);
#pragma unroll
    for (int k = 0; k < 5; ++k) Ut[k] += Q[k];
  }
  if (MODE == 0) {
    double* o = a.Ut + (size_t)e * 5 * n3 + v;
#pragma unroll
    for (int k = 0; k < 5; ++k) o[k * n3] = Ut[k];
  } else {
    const double dt = case_dt(a, ce);
    double* du = a.dU + (size_t)e * 5 * n3 + v;
    double* uo = a.Urk + (size_t)e * 5 * n3 + v;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double x = a.first_stage ? dt * Ut[k] : a.rkA * du[k * n3] + dt * Ut[k];
      du[k * n3] = x;
      uo[k * n3] = U[k] + a.rkB * x;
    }
  }
}

// ---------------------------------------------------------------------------
// Lifted gradients (Eq. lifting)
// ---------------------------------------------------------------------------
// shared memory: the tables (fixed point and FP64), the reduction words, then
// per element the q planes (4), two buffers of one direction's metric planes
// (2 x 3) and the sums (12), all padded node planes
template <int N>
struct LiftFix {
  using F = Fix<N>;
  static constexpr int h = F::n / 2;
  static constexpr int ntab = F::n % 2 == 0 ? 2 * h * h : F::n2;  // split table entries
  static constexpr int planes = 22;
  static constexpr int Q = 8, nred = F::W * Q + Q + 1;  // maxima: u, v, w, T, metrics by Cartesian component, ~T; flag
  static constexpr size_t head(int epb) { return (16 * ntab + 4 * (size_t)epb * nred + 15) & ~size_t(15); }
  static constexpr size_t bytes(int epb) { return head(epb) + 8 * (size_t)epb * planes * F::Pn; }
};

// Dhat split in shared memory: for even n its even and odd halves
template <int N>
__device__ __forceinline__ void lift_table_fx(const Ops* o, Fx* sD) {
  using L = LiftFix<N>;
  constexpr int h = L::h;
  for (int k = threadIdx.x; k < L::ntab; k += blockDim.x)
    sD[k] = Fix<N>::n % 2 == 0 ? fx_split(k < h * h ? o->fxHe[k] : o->fxHo[k - h * h]) : fx_split(o->fxH[k]);
}
// (u, v, w, T) of the element's nodes, in FP64, to the q planes, and the
// maxima of their magnitudes, of the metrics by Cartesian component and of T's
// complement (its minimum)
template <int N>
__device__ __forceinline__ void lift_prims_fx(const StageArgs& a, int e, long long* q, unsigned m[8], int t) {
  using F = Fix<N>;
  constexpr int n = F::n, n3 = F::n3, Pn = F::Pn;
  const double* Me = a.metric + (size_t)e * 10 * n3;
#pragma unroll
  for (int k = 0; k < 8; ++k) m[k] = 0;
  for (int v = t; v < n3; v += F::TPE) {
    double U[5];
    load_state64<n>(a, e, v, U);
    const Prim64 pr = prim64(U, a.gm1);
    const double T = pr.p * pr.ri * a.Rinv;
    double* qd = reinterpret_cast<double*>(q) + fx_pad<n>(v);
    qd[0] = pr.u, qd[Pn] = pr.v, qd[2 * Pn] = pr.w, qd[3 * Pn] = T;
    m[0] = max(m[0], fx_mag(pr.u)), m[1] = max(m[1], fx_mag(pr.v)), m[2] = max(m[2], fx_mag(pr.w));
    m[3] = max(m[3], fx_mag(T)), m[7] = max(m[7], ~fx_mag(T));
#pragma unroll
    for (int c = 0; c < 9; ++c) m[4 + c % 3] = max(m[4 + c % 3], fx_mag(Me[c * n3 + v]));
  }
}
// the temperature falls into quiet on a node's lines (sum_form); the velocity
// needs no such test: an error of 2^-60 of the element's largest gradient of a
// component is below FP64's rounding of the pressure in the momentum's sums
template <int N>
__device__ __forceinline__ bool lift_plain(bool bad, const unsigned* fin) {
  const bool ask = bad || ~fin[7] < fx_cut(fin[3]);
  __syncwarp();
  return !(blockDim.x == Fix<N>::TPE ? ask : __syncthreads_or(ask));
}
template <int N>
__device__ __forceinline__ SumForm lift_form(bool bad, const long long* q, const unsigned* fin, int t, unsigned* flag) {
  constexpr int n = Fix<N>::n;
  const unsigned cut = fx_cut(fin[3]);
  const double* T = reinterpret_cast<const double*>(q + 3 * Fix<N>::Pn);
  auto mag = [=](int v) { return fx_mag(T[fx_pad<n>(v)]); };
  return sum_form<N>(bad, t, flag, [=](int v) { return mag(v) < cut && lines_quiet<n>(v, cut, mag); });
}
// The volume sums sum_d Dhat (Ja^d q) of the element in the W planes, from the
// FP64 values in the q planes; a sum of variable k = 3 q + x has the scale
// 2^(fxH_bits - 2 - eq[q] - eJ[x]) and is below 2^62.  skip: an element whose
// sums are taken in FP64 (lift_sums_f64).
template <int N>
__device__ __forceinline__ void lift_sums_fx(const double* Me, long long* q, long long* J, long long* W, const Fx* sD,
                                             int t, const int eq[4], const int eJ[3], bool skip) {
  using F = Fix<N>;
  using L = LiftFix<N>;
  constexpr int n = F::n, n2 = F::n2, TPE = F::TPE, Pn = F::Pn, h = L::h;
  const int n3 = skip ? 0 : F::n3, tasks = skip ? 0 : 4 * n2;
  for (int v = t; v < n3; v += TPE) {
    const int pv = fx_pad<n>(v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      long long* x = q + k * Pn + pv;
      *x = fx_from<61>(__longlong_as_double(*x), eq[k]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) J[c * Pn + pv] = fx_from<60>(Me[c * F::n3 + v], eJ[c]);
  }
  __syncwarp();
  __syncthreads();
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const int sd = dir_stride<n>(d);
    const long long* Jd = J + (d & 1) * 3 * Pn;
    for (int task = t; task < tasks; task += TPE) {
      const int qv = task / n2, bl = line_base<n>(d, task % n2);
      Fx ql[n];
#pragma unroll
      for (int al = 0; al < n; ++al) ql[al] = fx_split(q[qv * Pn + fx_pad<n>(bl + al * sd)]);
#pragma unroll 1
      for (int x = 0; x < 3; ++x) {
        long long P[n];  // Ja^d_x q: |P| <= 2^(60 + 61 - 64 + 2)
#pragma unroll
        for (int al = 0; al < n; ++al) {
          FxSum<2> s;
          s.add(fx_split(Jd[x * Pn + fx_pad<n>(bl + al * sd)]), ql[al]);
          P[al] = s.get();
        }
        long long* w = W + (qv * 3 + x) * Pn;
        auto put = [&](int i, long long y) {
          long long* o = w + fx_pad<n>(bl + i * sd);
          *o = d == 0 ? y : *o + y;
        };
        // the rows of Dhat sum to at most 2^62: |y| <= 2^(62 + 59 - 64 + 3), three directions below 2^62
        if constexpr (n % 2 == 0) {
          // Dhat is centro-antisymmetric: even and odd halves (dg_types.h)
          Fx E[h], O[h];
#pragma unroll
          for (int j = 0; j < h; ++j) E[j] = fx_split(P[j] + P[n - 1 - j]), O[j] = fx_split(P[j] - P[n - 1 - j]);
#pragma unroll
          for (int i = 0; i < h; ++i) {
            FxSum<3> ev, od;
#pragma unroll
            for (int j = 0; j < h; ++j) ev.add(sD[i * h + j], E[j]), od.add(sD[h * h + i * h + j], O[j]);
            const long long ye = ev.get(), yo = od.get();
            put(i, yo + ye);
            put(n - 1 - i, yo - ye);
          }
        } else {
          Fx Ps[n];
#pragma unroll
          for (int j = 0; j < n; ++j) Ps[j] = fx_split(P[j]);
#pragma unroll
          for (int i = 0; i < n; ++i) {
            FxSum<3> s;
#pragma unroll
            for (int j = 0; j < n; ++j) s.add(sD[i * n + j], Ps[j]);
            put(i, s.get());
          }
        }
      }
    }
    if (d < 2) {  // the next direction's metrics into the other buffer
      long long* Jn = J + ((d + 1) & 1) * 3 * Pn;
      for (int v = t; v < n3; v += TPE)
#pragma unroll
        for (int c = 0; c < 3; ++c) Jn[c * Pn + fx_pad<n>(v)] = fx_from<60>(Me[(3 * d + 3 + c) * F::n3 + v], eJ[c]);
    }
    __syncwarp();
    __syncthreads();
  }
}
// the same in FP64, all planes holding FP64 values; sD: Dhat, for even n its
// even and odd halves
template <int N>
__device__ __forceinline__ void lift_sums_f64(const Ops* o, const double* Me, const double* q, double* J, double* W,
                                           double* sD, int t, bool skip) {
  using F = Fix<N>;
  using L = LiftFix<N>;
  constexpr int n = F::n, n2 = F::n2, TPE = F::TPE, Pn = F::Pn, h = L::h;
  const int n3 = skip ? 0 : F::n3, tasks = skip ? 0 : 4 * n2;
  for (int k = threadIdx.x; k < L::ntab; k += blockDim.x) {
    if constexpr (n % 2 == 0) {
      const double* D = o->Dhat + (k % (h * h)) / h * n;
      const int j = k % h;
      sD[k] = 0.5 * (k < h * h ? D[j] + D[n - 1 - j] : D[j] - D[n - 1 - j]);
    } else {
      sD[k] = o->Dhat[k];
    }
  }
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    double* Jd = J + (d & 1) * 3 * Pn;
    for (int v = t; v < n3; v += TPE)
#pragma unroll
      for (int c = 0; c < 3; ++c) Jd[c * Pn + fx_pad<n>(v)] = Me[(3 * d + c) * F::n3 + v];
    __syncwarp();
    __syncthreads();
    const int sd = dir_stride<n>(d);
    for (int task = t; task < tasks; task += TPE) {
      const int qv = task / n2, bl = line_base<n>(d, task % n2);
#pragma unroll 1
      for (int x = 0; x < 3; ++x) {
        double P[n];
#pragma unroll
        for (int al = 0; al < n; ++al) {
          const int pa = fx_pad<n>(bl + al * sd);
          P[al] = Jd[x * Pn + pa] * q[qv * Pn + pa];
        }
        double* w = W + (qv * 3 + x) * Pn;
        auto put = [&](int i, double y) {
          double* out = w + fx_pad<n>(bl + i * sd);
          *out = d == 0 ? y : *out + y;
        };
        if constexpr (n % 2 == 0) {
#pragma unroll
          for (int i = 0; i < h; ++i) {
            double ye = 0.0, yo = 0.0;
#pragma unroll
            for (int j = 0; j < h; ++j) {
              ye += sD[i * h + j] * (P[j] + P[n - 1 - j]);
              yo += sD[h * h + i * h + j] * (P[j] - P[n - 1 - j]);
            }
            put(i, yo + ye);
            put(n - 1 - i, yo - ye);
          }
        } else {
#pragma unroll
          for (int i = 0; i < n; ++i) {
            double y = 0.0;
#pragma unroll
            for (int j = 0; j < n; ++j) y += sD[i * n + j] * P[j];
            put(i, y);
          }
        }
      }
    }
    __syncwarp();
    __syncthreads();
  }
}

// the element's places in shared memory
template <int N>
struct LiftMem {
  using L = LiftFix<N>;
  Fx* sD;
  double* sDd;  // (filled by lift_sums_f64)
  unsigned *red, *fin, *flag;
  long long *q, *J, *W;  // [4][Pn], [2][3][Pn], [12][Pn]
  __device__ __forceinline__ LiftMem(unsigned char* smraw, int epb, int le) {
    sD = reinterpret_cast<Fx*>(smraw);
    sDd = reinterpret_cast<double*>(sD + L::ntab);
    red = reinterpret_cast<unsigned*>(smraw + 16 * L::ntab) + le * L::nred;
    fin = red + Fix<N>::W * L::Q;
    flag = fin + L::Q;
    q = reinterpret_cast<long long*>(smraw + L::head(epb)) + (size_t)le * L::planes * Fix<N>::Pn;
    J = q + 4 * Fix<N>::Pn;
    W = J + 6 * Fix<N>::Pn;
  }
};
template <int N>
__device__ __forceinline__ bool lift_bad(const unsigned* fin) {
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 7; ++k) bad = bad || fx_bad(fin[k]);
  return bad;
}
// the sums and what follows them; PLAIN: the block's elements are all in fixed point
template <int N, bool PLAIN>
__device__ __forceinline__ void lift_rest(const StageArgs& a, const LiftMem<N>& M, const ElemRef& er, int t) {
  using F = Fix<N>;
  constexpr int n = F::n, n2 = F::n2, n3 = F::n3, TPE = F::TPE, Pn = F::Pn;
  const int e = er.e;
  const double* Me = a.metric + (size_t)e * 10 * n3;
  const unsigned* fin = M.fin;
  const int eq[4] = {fx_exp(fin[0]), fx_exp(fin[1]), fx_exp(fin[2]), fx_exp(fin[3])};
  const int eJ[3] = {fx_exp(fin[4]), fx_exp(fin[5]), fx_exp(fin[6])};
  SumForm form = {false, false, false};
  if constexpr (!PLAIN) form = lift_form<N>(lift_bad<N>(fin), M.q, fin, t, M.flag);
  const bool bad = form.direct;
  if (!form.all) lift_sums_fx<N>(Me, M.q, M.J, M.W, M.sD, t, eq, eJ, bad);
  if (form.any)
    lift_sums_f64<N>(a.ops, Me, reinterpret_cast<const double*>(M.q), reinterpret_cast<double*>(M.J),
                     reinterpret_cast<double*>(M.W), M.sDd, t, !bad);
  if (!er.valid) return;
  const int pH = a.ops->fxH_bits - 2;
  const double* Lf = a.lflux;
  for (int v = t; v < n3; v += TPE) {
    const int pv = fx_pad<n>(v);
    double acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const long long w = M.W[k * Pn + pv];
      acc[k] = bad ? __longlong_as_double(w) : fx_to(w, pH - eq[k / 3] - eJ[k % 3]);
    }
    // surface part: on LGL nodes only face nodes receive it
    const int idx[3] = {v % n, (v / n) % n, v / n2};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int id = idx[d];
      if (id != 0 && id != n - 1) continue;
      const int f = 2 * d + (id == n - 1 ? 1 : 0);
      const int es = a.elem_side[(size_t)e * 6 + f];
      int p, qq;
      face_pq(d, idx, p, qq);
      int pm = p, qm = qq;
      if (es_slave(es)) flip_to_master<n>(es_flip(es), p, qq, pm, qm);
      const double sg = es_slave(es) ? -a.ops->winv[id] : a.ops->winv[id];
      const double* Lr = Lf + (size_t)es_side(es) * 12 * n2 + pm + n * qm;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] += sg * Lr[k * n2];
    }
    const double Ji = Me[9 * n3 + v];
    double* g = a.g + (size_t)e * 12 * n3 + v;
#pragma unroll
    for (int k = 0; k < 12; ++k) g[k * n3] = acc[k] * Ji;
  }
}

template <int N>
__device__ __noinline__ void lift_mixed(const StageArgs& a, ElemRef er) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / Fix<N>::TPE, le = threadIdx.x / Fix<N>::TPE;
  lift_rest<N, false>(a, LiftMem<N>(smraw, epb, le), er, threadIdx.x % Fix<N>::TPE);
}

template <int N>
__global__ void __launch_bounds__(Fix<N>::TL, Fix<N>::min_blocks(Fix<N>::TL)) k_lift_fx(const __grid_constant__ StageArgs a) {
  using F = Fix<N>;
  constexpr int TPE = F::TPE;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / TPE, le = threadIdx.x / TPE, t = threadIdx.x % TPE;
  const LiftMem<N> M(smraw, epb, le);
  const ElemRef er = elem_ref(a, blockIdx.x * epb + le);
  if (a.elem_case && __syncthreads_and(!er.busy)) return;
  lift_table_fx<N>(a.ops, M.sD);
  prefetch_sides64<N>(a, er.e, a.lflux, 12, t);
  prefetch_next64<N>(a, (blockIdx.x + a.prefetch) * epb + le, t - 32);
  if (t == 0) *M.flag = 0u;
  {
    unsigned m[8];
    lift_prims_fx<N>(a, er.e, M.q, m, t);
    fx_reduce<N, 8>(m, M.red, M.fin, t);
    __syncthreads();
  }
  if (lift_plain<N>(lift_bad<N>(M.fin), M.fin)) lift_rest<N, true>(a, M, er, t);
  else lift_mixed<N>(a, er);
}

// ---------------------------------------------------------------------------
// Volume integral + SurfInt + ApplyJac (+ RK update)
// ---------------------------------------------------------------------------
// Scales of an element's two-point sums, from its groups' maxima.  The metrics
// have an exponent eJ for each Cartesian component (over the three directions)
// and the velocity's component i is held as u_i 2^(eJ_i) under one exponent, so
// that the products u_i m_i of a stretched element meet in one scale.  For each
// direction the shifts bring every product's bound (from the actual maxima,
// component by component) next to 2^62, so that no bits go to loose bounds;
// the directions' sums are aligned at the end.
struct DirScale {
  int s1, s2, s3, s6;  // shifts of un, fr, t and energy (kep_flux_fx)
  // by momentum component: shift of the pressure (below zero: a right shift),
  // right shift of t (aligns it with the pressure), shift of the flux
  int s4[3], kc[3], s5[3];
  int aM, aV[3], aE;  // right shifts of the direction's mass, momentum and energy sums
};
struct VolScale {
  DirScale d[3];
  int eR, eP, eH, eU;  // eU: of the scaled velocity
  int eJ[3];
  int pM, pV[3], pE;   // results: sums times 2^-p
  int c[3][5];         // the directions' own scales
  unsigned bad, quiet, iso;
};
// maxima of magnitudes; VQ_LO: of the complements of density, pressure and rho H
// (their minima)
enum { VQ_RHO, VQ_U, VQ_V, VQ_W, VQ_P, VQ_H, VQ_RHOH, VQ_MOM, VQ_J, VQ_LO = VQ_J + 9, VQ_N = VQ_LO + 3 };

// Whether the predicate holds in any thread of the element's first warp (of
// the element, at N = 1), called by all of them
template <int N>
__device__ __forceinline__ bool fx_any(bool x, int t) {
  if constexpr (Fix<N>::TPE >= 32) return __any_sync(0xffffffffu, x);
  else return (__ballot_sync(0xffffffffu, x) >> ((threadIdx.x & 31) - t) & ((1u << Fix<N>::TPE) - 1u)) != 0u;
}
// a magnitude's logarithm to base two in units of 2^-20, at most 0.09 too small
// (its high word: exponent and fraction)
__device__ __forceinline__ int fx_log(unsigned mag) { return (int)mag - (1023 << 20); }

// Whether the element's two-point sums are in FP64 in any case: groups out of
// range, and elements whose largest fluxes lie far below the product of their
// groups' maxima (light and fast or hot fluid beside dense fluid, ratios above
// about four): their scale would leave the fluxes fewer bits than FP64 gives
// them.  Likewise a small velocity component beside fast flow: the error of
// t u_i is that of the largest component, below FP64's rounding of p m_i unless
// the dynamic pressure exceeds the pressure by far.  Threads of the first warp.
template <int N>
__device__ __forceinline__ bool vol_bad(const unsigned* m, int t) {
  bool bad = false;
  for (int k = t; k < VQ_LO; k += Fix<N>::TPE < 32 ? Fix<N>::TPE : 32) bad = bad || fx_bad(m[k]);
  const unsigned mu = max(max(m[VQ_U], m[VQ_V]), m[VQ_W]);
  const int r = fx_log(m[VQ_RHO]);
  if (t == 0) bad = bad || r + fx_log(m[VQ_H]) - fx_log(m[VQ_RHOH]) > 2 << 20;
  if (t == 1) bad = bad || (mu != 0u && r + fx_log(mu) - fx_log(m[VQ_MOM]) > 2 << 20);
  if (t >= 2 && t < 5) {
    const unsigned ui = m[VQ_U + t - 2];  // (unscaled: a stretched element's pressure terms differ as well)
    bad = bad || (ui != 0u && ui < fx_down(mu, 4) && r + 2 * fx_log(mu) - fx_log(m[VQ_P]) > 4 << 20);
  }
  return fx_any<N>(bad, t);
}

// Threads 0 .. 2 of the element form the shifts of one direction each
// (vol_scale) and then align the directions' sums (vol_align), which reads the
// other two threads' scales: the caller synchronises the whole warp between
// the two, outside the branch on the thread (at N = 1 it holds four elements).
// Returns whether the element is plain: the three components share their
// shifts (kep_fx) and no value is quiet or out of range.
__device__ __forceinline__ bool vol_scale(VolScale& s, const unsigned* m, const Ops* o, int t, bool bad) {
  const int eR = fx_exp(m[VQ_RHO]), eP = fx_exp(m[VQ_P]), eH = fx_exp(m[VQ_H]);
  int eJ[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) eJ[i] = fx_exp(max(max(m[VQ_J + i], m[VQ_J + 3 + i]), m[VQ_J + 6 + i]));
  const int eJx = max(max(eJ[0], eJ[1]), eJ[2]);
  // nearly equal components share the largest exponent (two bits at most)
  const bool iso = eJx - min(min(eJ[0], eJ[1]), eJ[2]) <= 2;
  if (iso) eJ[0] = eJ[1] = eJ[2] = eJx;
  const int eU = max(max(fx_exp(m[VQ_U]) + eJ[0], fx_exp(m[VQ_V]) + eJ[1]), fx_exp(m[VQ_W]) + eJ[2]);
  float uf[3], jf[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    uf[i] = fx_frac(m[VQ_U + i], eU - eJ[i]);
    jf[i] = fx_frac(m[VQ_J + 3 * t + i], eJ[i]);
  }
  const float fR = fx_frac(m[VQ_RHO], eR), fP = fx_frac(m[VQ_P], eP), fH = fx_frac(m[VQ_H], eH), fS = o->fxS_row;
  DirScale& d = s.d[t];
  // bounds in units of 2^58 (un), 2^60 and 2^61 (the others)
  float b = uf[0] * jf[0] + uf[1] * jf[1] + uf[2] * jf[2];
  const int s1 = fx_room(b, 4);
  b = fR * fx_scale(b, s1 - 4);  // fr / 2^60
  const int s2 = fx_room(b, 2);
  b = fS * fx_scale(b, s2 - 2);  // t / 2^60, summed over a row
  const int s3 = fx_room(b, 1);
  const float bt = fx_scale(b, s3 - 1);  // t / 2^61
  const float bp0 = fS * fP;             // pressure / 2^60
  const int s4 = fx_room(bp0, 2);
  d.s1 = s1, d.s2 = s2, d.s3 = s3;
  // scales: value times 2^a; the means' factors 1/8 (mass), 1/4 (pressure) and 1/16 (energy); 1/w (fxW)
  const int a3 = o->fxS_bits + 61 - eR + 56 - eU + s1 - 128 + s2 + s3;
  const int b3 = o->fxS_bits + 61 - eP - 64 + s4;
  const int w = o->fxW_bits - 62;
  s.c[t][0] = a3 + 3 + w;
  if (iso) uf[0] = fmaxf(uf[0], fmaxf(uf[1], uf[2])), jf[0] = fmaxf(jf[0], fmaxf(jf[1], jf[2]));
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (iso && i > 0) {  // as the first
      d.kc[i] = d.kc[0], d.s4[i] = d.s4[0], d.s5[i] = d.s5[0], s.c[t][1 + i] = s.c[t][1];
      continue;
    }
    // t u_i against p m_i; a component whose metric (or velocity) is zero has the other's scale
    const int at = a3 - (eU - eJ[i]) + 2, ap = b3 - eJ[i];
    const bool of_t = jf[i] == 0.0f || (at < ap && uf[i] != 0.0f);
    const int kc = of_t ? 0 : min(max(at - ap, 0), 62), kp = of_t ? min(max(ap - at, 0), 90) : 0;
    const float bp = jf[i] == 0.0f ? 0.0f : fx_scale(bp0, s4 - 1 - kp);  // pressure / 2^61
    const int s5 = fx_room(fx_scale(bt, -kc) * uf[i] + bp * jf[i], 3);  // momentum / 2^58
    d.kc[i] = kc;
    d.s4[i] = s4 - (jf[i] == 0.0f ? 90 : kp);
    d.s5[i] = s5;
    s.c[t][1 + i] = (of_t ? at : ap) - 2 + s5 + w;
  }
  d.s6 = fx_room(bt * fH, 2);  // energy / 2^59
  s.c[t][4] = a3 - eH + 1 + d.s6 + w;
  if (t == 0) {
    s.eR = eR, s.eU = eU, s.eP = eP, s.eH = eH;
#pragma unroll
    for (int i = 0; i < 3; ++i) s.eJ[i] = eJ[i];
    s.bad = bad;
    s.quiet = 0u;
    s.iso = iso;
  }
  return iso && !bad && ~m[VQ_LO] >= fx_cut(m[VQ_RHO]) && ~m[VQ_LO + 1] >= fx_cut(m[VQ_P]) &&
         ~m[VQ_LO + 2] >= fx_cut(m[VQ_RHOH]);
}
__device__ __forceinline__ void vol_align(VolScale& s, int t) {
  int p[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) p[k] = min(min(s.c[0][k], s.c[1][k]), s.c[2][k]);
  DirScale& d = s.d[t];
  d.aM = min(s.c[t][0] - p[0], 62), d.aE = min(s.c[t][4] - p[4], 62);
#pragma unroll
  for (int i = 0; i < 3; ++i) d.aV[i] = min(s.c[t][1 + i] - p[1 + i], 62);
  if (t == 0) {
    s.pM = p[0], s.pE = p[4];
#pragma unroll
    for (int i = 0; i < 3; ++i) s.pV[i] = p[1 + i];
  }
}
// The form of the element's two-point sums: in FP64 where the scales ask for
// it or where density, pressure or rho H are quiet on a node's lines (a corner
// of an element that a strong front just enters).  The velocity needs no such
// test: within a stable time step an error of 2^-59 of the element's largest
// mass or energy flux changes a node's density and energy by less than FP64's
// rounding of them (unless those are quiet), the momentum's by less than that
// of the pressure terms.
template <int N>
__device__ __forceinline__ SumForm vol_form(VolScale* sc, const unsigned* m, const longlong2* P, int t) {
  constexpr int n = Fix<N>::n, Pn = Fix<N>::Pn;
  const double2* Pd = reinterpret_cast<const double2*>(P);
  auto rho = [=](int v) { return fx_mag(Pd[fx_pad<n>(v)].x); };
  auto prs = [=](int v) { return fx_mag(Pd[fx_pad<n>(v)].y); };
  auto rhoH = [=](int v) { return fx_mag(Pd[fx_pad<n>(v)].x * Pd[2 * Pn + fx_pad<n>(v)].y); };
  const unsigned cR = fx_cut(m[VQ_RHO]), cP = fx_cut(m[VQ_P]), cH = fx_cut(m[VQ_RHOH]);
  return sum_form<N>(sc->bad != 0u, t, &sc->quiet, [=](int v) {
    return (rho(v) < cR && lines_quiet<n>(v, cR, rho)) || (prs(v) < cP && lines_quiet<n>(v, cP, prs)) ||
           (rhoH(v) < cH && lines_quiet<n>(v, cH, rhoH));
  });
}

// shared memory: S = w Dsplit, 1/w and Dhat split (Fx), Vinv, the reduction
// words and scales, then per element: the metrics (3 directions of (m0, m1)
// pairs and of m2), the primitives (pairs (rho, p), (u, v), (w, H)) and the
// two-point sums (5), all padded.  The viscous fluxes of one direction (pairs
// (f1, f2), (f3, f4), padded), the stress tensor and heat vector (9 planes,
// each thread's own nodes only) and the shock scratch take the place of the
// primitives and sums afterwards.
template <int N>
struct VolFix {
  using F = Fix<N>;
  static constexpr int offP = 9 * F::Pn;  // in 64-bit words
  static constexpr int offA = offP + 6 * F::Pn;
  static constexpr int offT = offP + 4 * F::Pn;  // after the viscous fluxes
  static constexpr int end1 = offA + 5 * F::Pn, end2 = offT + 9 * F::n3, end3 = offP + 2 * F::n3 + 4 * F::n2;
  static constexpr int end12 = end1 > end2 ? end1 : end2;
  static constexpr int per_elem = ((end12 > end3 ? end12 : end3) + 1) & ~1;
  static constexpr int nred = F::W * VQ_N + VQ_N;
  static constexpr int nscale = (int)(sizeof(VolScale) / 4);
  static constexpr int ntab = 3 * F::n2 + F::n;
  static constexpr size_t head(int epb) { return (8 * ntab + 4 * (size_t)epb * (nred + nscale) + 15) & ~size_t(15); }
  static constexpr size_t bytes(int epb) { return head(epb) + 8 * (size_t)epb * per_elem; }
  static_assert(offP % 2 == 0 && per_elem % 2 == 0 && (6 * F::Pn) % 2 == 0, "16-byte alignment of the pair planes");
};

// One two-point flux of KEP type, times S: (t, f1, f2, f3, f4).  ISO: the
// momentum components share their shifts.
struct KepNode {
  longlong2 a0, a1, a2, j0;  // (rho, p), (u, v), (w, H), (m0, m1)
  long long j1;              // m2
};
template <int n>
__device__ __forceinline__ KepNode kep_load(const longlong2* P, const longlong2* Jab, const long long* Jc, int pv) {
  constexpr int Pn = fx_plane<n>();
  return {P[pv], P[Pn + pv], P[2 * Pn + pv], Jab[pv], Jc[pv]};
}
template <bool ISO>
__device__ __forceinline__ void kep_flux_fx(const KepNode& x, const KepNode& y, Fx S, const DirScale& d, long long f[5]) {
  // sums of two values: u and m below 2^61, rho, p and H below 2^62; every
  // result below 2^62 by the choice of its shift
  const Fx m[3] = {fx_split(x.j0.x + y.j0.x), fx_split(x.j0.y + y.j0.y), fx_split(x.j1 + y.j1)};
  const Fx u[3] = {fx_split(x.a1.x + y.a1.x), fx_split(x.a1.y + y.a1.y), fx_split(x.a2.x + y.a2.x)};
  FxSumS un, fr, tt, f4;
  un.add(u[0], m[0]), un.add(u[1], m[1]), un.add(u[2], m[2]);
  fr.add(fx_split(x.a0.x + y.a0.x), fx_split(un.get(d.s1)));
  tt.add(S, fx_split(fr.get(d.s2)));
  f[0] = tt.get(d.s3);
  const Fx p = fx_split(x.a0.y + y.a0.y);
  Fx tk, ps;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (!ISO || i == 0) {
      const int s4 = d.s4[i];
      FxSumS pd;
      pd.add(S, p);
      tk = fx_split(f[0] >> d.kc[i]);
      ps = fx_split(s4 >= 0 ? pd.get(s4) : pd.get(0) >> min(-s4, 62));
    }
    FxSumS fi;
    fi.add(tk, u[i]), fi.add(ps, m[i]);
    f[1 + i] = fi.get(d.s5[ISO ? 0 : i]);
  }
  f4.add(fx_split(f[0]), fx_split(x.a2.y + y.a2.y));
  f[4] = f4.get(d.s6);
}

// Split-form KEP sums of all nodes: each thread takes one node of a line that
// its warp holds whole, forms the fluxes to the partners 1 .. (n - 1) / 2
// places on (cyclically), adds them to its own sums and passes them to the
// partner, whose S has the opposite sign (S = w Dsplit is antisymmetric); for
// even n the partner n / 2 places on is taken from both sides.  That is 3 + 1
// fluxes per node and direction at n = 8 where every node summing over all
// its partners takes 7.
template <int N, bool ISO>
__device__ __forceinline__ void kep_fx(const longlong2* P, const longlong2* Jab, const long long* Jc, long long* A,
                                       const Fx* sS, const Fx* sW, const VolScale* sc, int t, bool skip) {
  using F = Fix<N>;
  constexpr int n = F::n, n3 = F::n3, Pn = F::Pn, LW = F::LW;
  const int lane = F::TPE >= 32 ? t & 31 : t;
  const int lane0 = F::TPE >= 32 ? 0 : (threadIdx.x & 31) - t;  // the element's first lane
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const DirScale ds = sc->d[d];
    const int sd = dir_stride<n>(d);
    const longlong2* Jd = Jab + d * Pn;
    const long long* Jcd = Jc + d * Pn;
#pragma unroll 1
    for (int r = 0; r < F::RL; ++r) {
      const int slot = ((t / 32) + r * F::W) * LW + lane;
      const bool on = lane < LW && slot < n3 && !skip;
      const int line = on ? slot / n : 0, id = lane % n, base = line_base<n>(d, line);
      const int pv = fx_pad<n>(base + id * sd);
      long long acc[5] = {0, 0, 0, 0, 0};
      const KepNode me = kep_load<n>(P, Jd, Jcd, pv);
#pragma unroll 1
      for (int k = 1; k <= (n - 1) / 2; ++k) {
        const int al = id + k < n ? id + k : id + k - n, from = id >= k ? id - k : id - k + n;
        long long f[5];
        kep_flux_fx<ISO>(me, kep_load<n>(P, Jd, Jcd, fx_pad<n>(base + al * sd)), sS[id * n + al], ds, f);
        const int src = min(lane0 + lane - id + from, 31);
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[c] += f[c] - __shfl_sync(0xffffffffu, f[c], src);
      }
      if constexpr (n % 2 == 0) {
        const bool low = id < n / 2;  // (S of the lower node, so that both take the same flux)
        const int al = low ? id + n / 2 : id - n / 2;
        long long f[5];
        kep_flux_fx<ISO>(me, kep_load<n>(P, Jd, Jcd, fx_pad<n>(base + al * sd)), sS[min(id, al) * n + max(id, al)], ds, f);
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[c] += low ? f[c] : -f[c];
      }
      if (on) {
        const Fx wi = sW[id];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          FxSum<2> y;  // 2^(61 + 62 - 64 + 2)
          y.add(wi, fx_split(acc[c]));
          const long long z = fx_shr(y.get(), c == 0 ? ds.aM : c == 4 ? ds.aE : ds.aV[ISO ? 0 : c - 1]);
          A[c * Pn + pv] = d == 0 ? z : A[c * Pn + pv] + z;
        }
      }
    }
    __syncwarp();
    __syncthreads();
  }
}
// the same in FP64 (P, J and A hold FP64 values), with the same exchange of
// fluxes, so that an element whose sums are taken here costs the FP64 unit as
// many of them
template <int N>
__device__ __forceinline__ void kep_f64(const double2* P, const double2* Jab, const double* Jc, double* A,
                                     const double* Dsplit, int t, bool skip) {
  using F = Fix<N>;
  constexpr int n = F::n, n3 = F::n3, Pn = F::Pn, LW = F::LW;
  const int lane = F::TPE >= 32 ? t & 31 : t;
  const int lane0 = F::TPE >= 32 ? 0 : (threadIdx.x & 31) - t;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const int sd = dir_stride<n>(d);
    const double2* Jd = Jab + d * Pn;
    const double* Jcd = Jc + d * Pn;
#pragma unroll 1
    for (int r = 0; r < F::RL; ++r) {
      const int slot = ((t / 32) + r * F::W) * LW + lane;
      const bool on = lane < LW && slot < n3 && !skip;
      const int line = on ? slot / n : 0, id = lane % n, base = line_base<n>(d, line);
      const int pv = fx_pad<n>(base + id * sd);
      const double2 a0 = P[pv], a1 = P[Pn + pv], a2 = P[2 * Pn + pv], j0 = Jd[pv];
      const double j1 = Jcd[pv];
      double acc[5] = {0, 0, 0, 0, 0};
      auto flux = [&](int al, double f[5]) {  // eight times the flux's mass part, and so on
        const int pa = fx_pad<n>(base + al * sd);
        const double2 b0 = P[pa], b1 = P[Pn + pa], b2 = P[2 * Pn + pa], c0 = Jd[pa];
        const double m0 = j0.x + c0.x, m1 = j0.y + c0.y, m2 = j1 + Jcd[pa];  // twice the means
        const double u0 = a1.x + b1.x, u1 = a1.y + b1.y, u2 = a2.x + b2.x, p = 2.0 * (a0.y + b0.y);
        const double fr = (a0.x + b0.x) * (u0 * m0 + u1 * m1 + u2 * m2), hf = 0.5 * fr;
        f[0] = fr, f[1] = hf * u0 + p * m0, f[2] = hf * u1 + p * m1, f[3] = hf * u2 + p * m2, f[4] = hf * (a2.y + b2.y);
      };
      double f[5];
#pragma unroll
      for (int k = 1; k <= (n - 1) / 2; ++k) {
        const int al = id + k < n ? id + k : id + k - n, from = id >= k ? id - k : id - k + n;
        flux(al, f);
        const int src = min(lane0 + lane - id + from, 31);
        const double D = 0.125 * Dsplit[id * n + al], Df = 0.125 * Dsplit[id * n + from];
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[c] += D * f[c] + Df * __shfl_sync(0xffffffffu, f[c], src);
      }
      if constexpr (n % 2 == 0) {
        const int al = id < n / 2 ? id + n / 2 : id - n / 2;
        const double D = 0.125 * Dsplit[id * n + al];
        flux(al, f);
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[c] += D * f[c];
      }
      if (on) {
#pragma unroll
        for (int c = 0; c < 5; ++c) A[c * Pn + pv] = d == 0 ? acc[c] : A[c * Pn + pv] + acc[c];
      }
    }
    __syncwarp();
    __syncthreads();
  }
}

// the element's places in shared memory
template <int N>
struct VolMem {
  using L = VolFix<N>;
  Fx *sS, *sDh, *sW;  // [n2] w Dsplit, [n2] Dhat, [n] 1 / w
  double* sVi;        // [n2]
  unsigned *red, *fin;
  VolScale* sc;
  longlong2* Jab;  // [3][Pn] (m0, m1)
  long long* Jc;   // [3][Pn] m2
  long long* PT;   // the primitives' place
  long long* A;    // [5][Pn]
  __device__ __forceinline__ VolMem(unsigned char* smraw, int epb, int le) {
    constexpr int n = Fix<N>::n, n2 = Fix<N>::n2, Pn = Fix<N>::Pn;
    sS = reinterpret_cast<Fx*>(smraw);
    sDh = sS + n2;
    sW = sDh + n2;
    sVi = reinterpret_cast<double*>(sW + n);
    red = reinterpret_cast<unsigned*>(sVi + n2) + le * (L::nred + L::nscale);
    fin = red + Fix<N>::W * VQ_N;
    sc = reinterpret_cast<VolScale*>(fin + VQ_N);
    long long* mine = reinterpret_cast<long long*>(smraw + L::head(epb)) + (size_t)le * L::per_elem;
    Jab = reinterpret_cast<longlong2*>(mine);
    Jc = mine + 6 * Pn;
    PT = mine + L::offP;
    A = mine + L::offA;
  }
};
// What follows the scales.  EXTRA: a run with shock capturing, a sponge or a
// source; PLAIN: the block's elements are all plain (vol_scale).
template <int N, int MODE, bool EXTRA, bool PLAIN>
__device__ __forceinline__ void vol_rest(const StageArgs& a, const VolMem<N>& M, const ElemRef& er, const CaseParams& cp, int t) {
  using F = Fix<N>;
  using L = VolFix<N>;
  constexpr int n = F::n, n2 = F::n2, n3 = F::n3, TPE = F::TPE, Pn = F::Pn, R = F::R;
  const Fx *sS = M.sS, *sDh = M.sDh, *sW = M.sW;
  const double* sVi = M.sVi;
  unsigned *red = M.red, *fin = M.fin;
  VolScale* sc = M.sc;
  longlong2 *Jab = M.Jab, *P = reinterpret_cast<longlong2*>(M.PT);  // P: [3][Pn]
  long long *Jc = M.Jc, *PT = M.PT, *A = M.A, *mine = reinterpret_cast<long long*>(M.Jab);
  longlong2* G = P;  // [2][Pn] (after the two-point sums)
  const int e = er.e;
  const double* Me = a.metric + (size_t)e * 10 * n3;
  bool iso = true;
  SumForm form = {false, false, false};
  if constexpr (!PLAIN) {
    iso = __syncthreads_and(sc->iso != 0u);
    form = vol_form<N>(sc, fin, P, t);
  }
  const bool bad = form.direct;
  for (int v = t; v < n3; v += TPE) {
    const int pv = fx_pad<n>(v);
    double mt[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) mt[c] = Me[c * n3 + v];
    if (bad) {  // FP64 values
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        reinterpret_cast<double2*>(Jab)[d * Pn + pv] = make_double2(mt[3 * d], mt[3 * d + 1]);
        reinterpret_cast<double*>(Jc)[d * Pn + pv] = mt[3 * d + 2];
      }
    } else {
      const double2* Pd = reinterpret_cast<const double2*>(P) + pv;
      const double2 x0 = Pd[0], x1 = Pd[Pn], x2 = Pd[2 * Pn];
      P[pv] = make_longlong2(fx_from<61>(x0.x, sc->eR), fx_from<61>(x0.y, sc->eP));
      const int e0 = sc->eJ[0], e1 = sc->eJ[1], e2 = sc->eJ[2], eU = sc->eU;
      P[Pn + pv] = make_longlong2(fx_from<60>(x1.x, eU - e0), fx_from<60>(x1.y, eU - e1));
      P[2 * Pn + pv] = make_longlong2(fx_from<60>(x2.x, eU - e2), fx_from<61>(x2.y, sc->eH));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        Jab[d * Pn + pv] = make_longlong2(fx_from<60>(mt[3 * d], e0), fx_from<60>(mt[3 * d + 1], e1));
        Jc[d * Pn + pv] = fx_from<60>(mt[3 * d + 2], e2);
      }
    }
  }
  __syncwarp();
  __syncthreads();
  // ---- split-form KEP volume integral ----
  if (!form.all) {
    if (iso) kep_fx<N, true>(P, Jab, Jc, A, sS, sW, sc, t, bad);
    else kep_fx<N, false>(P, Jab, Jc, A, sS, sW, sc, t, bad);
  }
  if (form.any)
    kep_f64<N>(reinterpret_cast<const double2*>(P), reinterpret_cast<const double2*>(Jab),
               reinterpret_cast<const double*>(Jc), reinterpret_cast<double*>(A), a.ops->Dsplit, t, !bad);
  double conv[R][5];  // convective DG volume term
  double visc[R][4];  // viscous volume term
  long long vel[R][3];  // the velocity in fixed point (FP64 values in a bad element)
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int v = t + r * TPE, pv = fx_pad<n>(v < n3 ? v : 0);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const long long y = A[k * Pn + pv];
      conv[r][k] = bad ? __longlong_as_double(y) : fx_to(y, k == 0 ? sc->pM : k == 4 ? sc->pE : sc->pV[k - 1]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) visc[r][k] = 0.0;
    vel[r][0] = P[Pn + pv].x, vel[r][1] = P[Pn + pv].y, vel[r][2] = P[2 * Pn + pv].x;
  }
  __syncwarp();
  __syncthreads();  // the primitives' and sums' planes are free
  // ---- viscous volume term: collocated weak form, per direction ----
  if (a.viscous) {
    // [9][n3]: tau and lambda grad T, then tau and W = tau u + lambda grad T
    // (the work term in fixed point: 19 FP64 operations less per node); each
    // thread reads back its own nodes only
    long long* T = mine + L::offT;
    {
      unsigned mv[4] = {0, 0, 0, 0};
      for (int v = t; v < n3; v += TPE) {
        double g[12];
        const double* pg = a.g + (size_t)e * 12 * n3 + v;
#pragma unroll
        for (int k = 0; k < 12; ++k) g[k] = pg[k * n3];
        double vmu, vlam, Tt = 0.0;
        if (a.sutherland) {
          double U[5];
          load_state64<n>(a, e, v, U);
          const Prim64 pr = prim64(U, a.gm1);
          Tt = pr.p * pr.ri * a.Rinv;
        }
        visc_coeffs<double>(a, cp, Tt, vmu, vlam);
        const double tw = (2.0 / 3.0) * (g[0] + g[4] + g[8]);
        const double x[9] = {vmu * (2.0 * g[0] - tw), vmu * (2.0 * g[4] - tw), vmu * (2.0 * g[8] - tw),
                             vmu * (g[1] + g[3]),     vmu * (g[2] + g[6]),     vmu * (g[5] + g[7]),
                             vlam * g[9],             vlam * g[10],            vlam * g[11]};
        double* Td = reinterpret_cast<double*>(T) + v;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          Td[k * n3] = x[k];
          mv[k < 6 ? 0 : k - 5] = max(mv[k < 6 ? 0 : k - 5], fx_mag(x[k]));
        }
      }
      fx_reduce<N, 4>(mv, red, fin, t);
      __syncthreads();
    }
    // The six stresses share an exponent and are contracted with the metrics
    // at their largest component's: an error below FP64's rounding of the
    // pressure terms of the same sums while the stresses stay below the
    // pressure by the element's stretching.  W_j is held as W_j 2^(eJ_j), like
    // the velocity.  (An element that leaves the range only here has its
    // metrics in fixed point: the FP64 sums then read them from memory.)
    const int eJ[3] = {sc->eJ[0], sc->eJ[1], sc->eJ[2]};
    const int eJm = max(max(eJ[0], eJ[1]), eJ[2]), eJn = min(min(eJ[0], eJ[1]), eJ[2]);
    const int eT = fx_exp(fin[0]), eL[3] = {fx_exp(fin[1]), fx_exp(fin[2]), fx_exp(fin[3])};
    const bool vbad = bad || fx_bad(fin[0]) || fx_bad(fin[1]) || fx_bad(fin[2]) || fx_bad(fin[3]) ||
                      eT + eJm - eJn > sc->eP + 1;
    const int eUm = sc->eU - eJn, eTU = eT + eUm;
    // W_j: below 2^60 at 2^(60 - eW + eJ_j)
    const int eW = max(max(max(eTU, eL[0]) + eJ[0], max(eTU, eL[1]) + eJ[1]), max(eTU, eL[2]) + eJ[2]) + 2;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int v = t + r * TPE;
      if (v >= n3) break;
      if (vbad) {
        double u[3];
        if (bad) {
#pragma unroll
          for (int k = 0; k < 3; ++k) u[k] = __longlong_as_double(vel[r][k]);
        } else {
#pragma unroll
          for (int k = 0; k < 3; ++k) u[k] = fx_to(vel[r][k], 60 - sc->eU + eJ[k]);
        }
        double* Td = reinterpret_cast<double*>(T) + v;
        const double t0 = Td[0], t1 = Td[n3], t2 = Td[2 * n3], t3 = Td[3 * n3], t4 = Td[4 * n3], t5 = Td[5 * n3];
        Td[6 * n3] = t0 * u[0] + t3 * u[1] + t4 * u[2] + Td[6 * n3];
        Td[7 * n3] = t3 * u[0] + t1 * u[1] + t5 * u[2] + Td[7 * n3];
        Td[8 * n3] = t4 * u[0] + t5 * u[1] + t2 * u[2] + Td[8 * n3];
      } else {
        Fx x[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const long long q = fx_from<60>(__longlong_as_double(T[k * n3 + v]), eT);
          T[k * n3 + v] = q;
          x[k] = fx_split(q);
        }
        const Fx u = fx_split(fx_shr(vel[r][0], min(eJ[0] - eJn, 62))), w1 = fx_split(fx_shr(vel[r][1], min(eJ[1] - eJn, 62))),
                 w2 = fx_split(fx_shr(vel[r][2], min(eJ[2] - eJn, 62)));
        FxSum<2> w[3];  // 3 2^(60 + 60 - 64 + 2) < 2^59.6
        w[0].add(x[0], u), w[0].add(x[3], w1), w[0].add(x[4], w2);
        w[1].add(x[3], u), w[1].add(x[1], w1), w[1].add(x[5], w2);
        w[2].add(x[4], u), w[2].add(x[5], w1), w[2].add(x[2], w2);
#pragma unroll
        for (int k = 0; k < 3; ++k)
          T[(6 + k) * n3 + v] = fx_shr(w[k].get(), min(eW - eJ[k] - 2 - eTU, 62)) +
                                fx_shr(fx_from<58>(__longlong_as_double(T[(6 + k) * n3 + v]), eL[k]), min(eW - eJ[k] - 2 - eL[k], 62));
      }
    }
    long long acc[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[r][k] = 0;
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
      for (int v = t; v < n3; v += TPE) {
        const int pv = fx_pad<n>(v);
        if (vbad) {
          const double* Td = reinterpret_cast<const double*>(T) + v;
          double tau[6], W[3], fv[4];
          const double nv[3] = {Me[3 * d * n3 + v], Me[(3 * d + 1) * n3 + v], Me[(3 * d + 2) * n3 + v]};
#pragma unroll
          for (int k = 0; k < 6; ++k) tau[k] = Td[k * n3];
#pragma unroll
          for (int k = 0; k < 3; ++k) W[k] = Td[(6 + k) * n3];
          viscous_flux_n(tau, W, nv, fv);
          reinterpret_cast<double2*>(G)[pv] = make_double2(fv[0], fv[1]);
          reinterpret_cast<double2*>(G)[Pn + pv] = make_double2(fv[2], fv[3]);
        } else {
          const longlong2 jab = Jab[d * Pn + pv];
          const long long jc = Jc[d * Pn + pv];
          const Fx c0 = fx_split(jab.x), c1 = fx_split(jab.y), c2 = fx_split(jc);  // by component, for W
          Fx j0 = c0, j1 = c1, j2 = c2;                                           // at the largest's exponent
          if (!iso)
            j0 = fx_split(fx_shr(jab.x, min(eJm - eJ[0], 62))), j1 = fx_split(fx_shr(jab.y, min(eJm - eJ[1], 62))),
            j2 = fx_split(fx_shr(jc, min(eJm - eJ[2], 62)));
          Fx x[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) x[k] = fx_split(T[k * n3 + v]);
          FxSum<2> f1, f2, f3, f4;  // 3 2^(60 + 60 - 64 + 2) < 2^59.6
          f1.add(x[0], j0), f1.add(x[3], j1), f1.add(x[4], j2);
          f2.add(x[3], j0), f2.add(x[1], j1), f2.add(x[5], j2);
          f3.add(x[4], j0), f3.add(x[5], j1), f3.add(x[2], j2);
          f4.add(x[6], c0), f4.add(x[7], c1), f4.add(x[8], c2);
          G[pv] = make_longlong2(f1.get(), f2.get());
          G[Pn + pv] = make_longlong2(f3.get(), f4.get());
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
          if (vbad) {
            const double2* Gd = reinterpret_cast<const double2*>(G);
            for (int al = 0; al < n; ++al) {
              const double c = a.ops->Dhat[id * n + al];
              const double2 g0 = Gd[fx_pad<n>(base + al * sd)], g1 = Gd[Pn + fx_pad<n>(base + al * sd)];
              visc[r][0] += c * g0.x, visc[r][1] += c * g0.y, visc[r][2] += c * g1.x, visc[r][3] += c * g1.y;
            }
          } else {
            FxSum<3> s1, s2, s3, s4;  // 2^(62 + 59.6 - 64 + 3) per direction
#pragma unroll
            for (int al = 0; al < n; ++al) {
              const int pa = fx_pad<n>(base + al * sd);
              const longlong2 g0 = G[pa], g1 = G[Pn + pa];
              const Fx c = sDh[id * n + al];
              s1.add(c, fx_split(g0.x)), s2.add(c, fx_split(g0.y)), s3.add(c, fx_split(g1.x)), s4.add(c, fx_split(g1.y));
            }
            acc[r][0] += s1.get(), acc[r][1] += s2.get(), acc[r][2] += s3.get(), acc[r][3] += s4.get();
          }
        }
      }
      __syncwarp();
      __syncthreads();
    }
    const int pT = a.ops->fxH_bits - 3 - eT - eJm, pW = a.ops->fxH_bits - 3 - eW;
    if (!vbad) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < 4; ++k) visc[r][k] = fx_to(acc[r][k], k < 3 ? pT : pW);
    }
  }
  // ---- shock capturing: indicator and FV sub-cell blending (Sec. 2.3) ----
  if (EXTRA && a.shock) {
    double al;
    if (a.alpha_force >= 0) {
      al = a.alpha_force;
    } else {
      double* X1 = reinterpret_cast<double*>(PT);
      for (int v = t; v < n3; v += TPE) {
        double U[5];
        load_state64<n>(a, e, v, U);
        X1[v] = U[0] * prim64(U, a.gm1).p;
      }
      al = element_alpha<n, TPE>(X1, X1 + n3, X1 + 2 * n3, sVi, a.ops, t, a.alpha_min, a.alpha_max);
    }
    if (er.valid && t == 0) a.alpha[e] = al;
    // block-uniform condition: the FV pass has barriers, and the elements of
    // one block may have different blending factors
    if (__syncthreads_or(al > 0)) {
      double* Gf = reinterpret_cast<double*>(PT);  // [5][n3]
      double vfv[R][5];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < 5; ++k) vfv[r][k] = 0.0;
      const double* FVm = a.fvmetric + (size_t)e * 3 * (n - 1) * 3 * n2;
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int sd = dir_stride<n>(d);
        // the flux through interface id + 1/2 is formed by the node on its left
        for (int v = t; v < n3; v += TPE) {
          const int id = dir_index<n>(v, d);
          if (id == n - 1) continue;
          const int idx[3] = {v % n, (v / n) % n, v / n2};
          const int line = d == 0 ? idx[1] + n * idx[2] : (d == 1 ? idx[0] + n * idx[2] : idx[0] + n * idx[1]);
          const double* fm = FVm + (size_t)(d * (n - 1) + id) * 3 * n2 + line;
          const double mv[3] = {fm[0], fm[n2], fm[2 * n2]};
          const double sAd = sqrt(mv[0] * mv[0] + mv[1] * mv[1] + mv[2] * mv[2]);
          const double sAi = 1.0 / sAd;
          const double nu[3] = {mv[0] * sAi, mv[1] * sAi, mv[2] * sAi};
          double UL[5], UR[5], fb[5];
          load_state64<n>(a, e, v, UL);
          load_state64<n>(a, e, v + sd, UR);
          lf_flux_s(shifted_prim<double>(UL, a.gm1, a.Rinv, cp), shifted_prim<double>(UR, a.gm1, a.Rinv, cp), nu,
                    a.gamma, cp.pr, fb);
#pragma unroll
          for (int k = 0; k < 5; ++k) Gf[k * n3 + v] = fb[k] * sAd;
        }
        __syncwarp();
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int v = t + r * TPE;
          if (v < n3) {
            const int id = dir_index<n>(v, d);
            const double wi = a.ops->winv[id];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
              if (id < n - 1) vfv[r][k] += Gf[k * n3 + v] * wi;
              if (id > 0) vfv[r][k] -= Gf[k * n3 + v - sd] * wi;
            }
          }
        }
        __syncwarp();
        __syncthreads();
      }
      if (al > 0) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int k = 0; k < 5; ++k) conv[r][k] = (1 - al) * conv[r][k] + al * vfv[r][k];
      }
    }
  }
  if (!er.valid) return;
  // a serving case that finished or sits this step out keeps its state
  if (MODE == 1 && !er.busy) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int v = t + r * TPE;
    if (v >= n3) break;
    double s[5] = {conv[r][0], conv[r][1] - visc[r][0], conv[r][2] - visc[r][1], conv[r][3] - visc[r][2],
                   conv[r][4] - visc[r][3]};
    // ---- SurfInt: face nodes receive +-f* lhat ----
    const int idx[3] = {v % n, (v / n) % n, v / n2};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int id = idx[d];
      if (id != 0 && id != n - 1) continue;
      const int f = 2 * d + (id == n - 1 ? 1 : 0);
      const int es = a.elem_side[(size_t)e * 6 + f];
      int p, qq;
      face_pq(d, idx, p, qq);
      int pm = p, qm = qq;
      if (es_slave(es)) flip_to_master<n>(es_flip(es), p, qq, pm, qm);
      const double sg = es_slave(es) ? -a.ops->winv[id] : a.ops->winv[id];
      const double* Fs = a.fstar + (size_t)es_side(es) * 5 * n2 + pm + n * qm;
#pragma unroll
      for (int k = 0; k < 5; ++k) s[k] += sg * Fs[k * n2];
    }
    finish_node64<n, MODE, EXTRA>(a, e, er.ce, v, s);
  }
}
template <int N, int MODE, bool EXTRA>
__device__ __noinline__ void vol_mixed(const StageArgs& a, ElemRef er) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / Fix<N>::TPE, le = threadIdx.x / Fix<N>::TPE;
  vol_rest<N, MODE, EXTRA, false>(a, VolMem<N>(smraw, epb, le), er, case_params(a, er.ce), threadIdx.x % Fix<N>::TPE);
}

template <int N, int MODE, bool EXTRA>
__global__ void __launch_bounds__(Fix<N>::TV, Fix<N>::min_blocks(Fix<N>::TV))
    k_volume_fx(const __grid_constant__ StageArgs a) {
  using F = Fix<N>;
  constexpr int n = F::n, n2 = F::n2, n3 = F::n3, TPE = F::TPE, Pn = F::Pn;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int epb = blockDim.x / TPE, le = threadIdx.x / TPE, t = threadIdx.x % TPE;
  const VolMem<N> M(smraw, epb, le);
  longlong2* P = reinterpret_cast<longlong2*>(M.PT);
  const ElemRef er = elem_ref(a, blockIdx.x * epb + le);
  if (a.elem_case && __syncthreads_and(!er.busy)) return;
  const int e = er.e;
  const CaseParams cp = case_params(a, er.ce);
  const double* Me = a.metric + (size_t)e * 10 * n3;
  for (int k = threadIdx.x; k < n2; k += blockDim.x) {
    M.sS[k] = fx_split(a.ops->fxS[k]);
    M.sDh[k] = fx_split(a.ops->fxH[k]);
    M.sVi[k] = a.ops->Vinv[k];
    if (k < n) M.sW[k] = fx_split(a.ops->fxW[k]);
  }
  prefetch_sides64<N>(a, e, a.fstar, 5, t);
  if (t == 6 && a.viscous) prefetch64(a.g, (size_t)e * 12 * n3, 12 * n3);
  if (t == 7 && MODE == 1 && !a.first_stage) prefetch64(a.dU, (size_t)e * 5 * n3, 5 * n3);
  prefetch_next64<N>(a, (blockIdx.x + a.prefetch) * epb + le, t - 32);
  // ---- primitives (FP64 in their planes until the scales are known), maxima ----
  bool plain = true;
  {
    unsigned m[VQ_N];
#pragma unroll
    for (int k = 0; k < VQ_N; ++k) m[k] = 0;
    for (int v = t; v < n3; v += TPE) {
      double U[5];
      load_state64<n>(a, e, v, U);
      const Prim64 pr = prim64(U, a.gm1);
      const double rH = U[4] + pr.p, H = rH * pr.ri;
      double2* Pd = reinterpret_cast<double2*>(P) + fx_pad<n>(v);
      Pd[0] = make_double2(pr.rho, pr.p);
      Pd[Pn] = make_double2(pr.u, pr.v);
      Pd[2 * Pn] = make_double2(pr.w, H);
      m[VQ_RHO] = max(m[VQ_RHO], fx_mag(pr.rho)), m[VQ_LO] = max(m[VQ_LO], ~fx_mag(pr.rho));
      m[VQ_U] = max(m[VQ_U], fx_mag(pr.u));
      m[VQ_V] = max(m[VQ_V], fx_mag(pr.v));
      m[VQ_W] = max(m[VQ_W], fx_mag(pr.w));
      m[VQ_P] = max(m[VQ_P], fx_mag(pr.p)), m[VQ_LO + 1] = max(m[VQ_LO + 1], ~fx_mag(pr.p));
      m[VQ_H] = max(m[VQ_H], fx_mag(H));
      m[VQ_RHOH] = max(m[VQ_RHOH], fx_mag(rH)), m[VQ_LO + 2] = max(m[VQ_LO + 2], ~fx_mag(rH));
      m[VQ_MOM] = max(max(m[VQ_MOM], fx_mag(U[1])), max(fx_mag(U[2]), fx_mag(U[3])));
#pragma unroll
      for (int c = 0; c < 9; ++c) m[VQ_J + c] = max(m[VQ_J + c], fx_mag(Me[c * n3 + v]));
    }
    fx_reduce<N, VQ_N>(m, M.red, M.fin, t);
    bool out = false;
    if (t < 32) out = a.sums64 || vol_bad<N>(M.fin, t);
    if (t < 3) plain = vol_scale(*M.sc, M.fin, a.ops, t, out);
    __syncwarp();
    if (t < 3) vol_align(*M.sc, t);
    __syncwarp();
    plain = __syncthreads_and(plain);  // (all of the block's elements)
  }
  if (plain) vol_rest<N, MODE, EXTRA, true>(a, M, er, cp, t);
  else vol_mixed<N, MODE, EXTRA>(a, er);
}

}  // namespace dg

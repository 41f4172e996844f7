// dpr1_arrow.cu -- eigenpairs of a real symmetric arrowhead matrix A = [D z; z^T alpha] of
// order n + 1 (D = diag(d), d strictly decreasing, no zero weight), the companion problem the
// paper relates its method to (Sec. 1), by the steps of Algorithm 1 on the shifted inverse.
//
// The eigenvalues interlace the poles, lambda_0 > d_0 > lambda_1 > ... > d_{n-1} > lambda_n,
// and are the zeros of f(lambda) = alpha - lambda - sum_j zeta_j^2 / (d_j - lambda), which
// decreases between consecutive poles.  Eigenvalue k is computed at the nearer pole d_i of
// its interval (lambda_0 at d_0, lambda_n at d_{n-1}; otherwise the sign of f at the
// midpoint decides).  (A - d_i I)^{-1} is again an arrowhead: with Delta_j = d_j - d_i its
// diagonal is 1/Delta_j (j != i), b at position i and 0 at position n; its border is
// w_j = -zeta_j / (zeta_i Delta_j) and 1/zeta_i at position n, and
//   b = (1/zeta_i^2) (sum_{j != i} zeta_j^2 / Delta_j - (alpha - d_i))
// is the DPR1 corner of Eq. (b_ob) with 1/rho replaced by d_i - alpha (double-double).  Its
// secular function is the DPR1 one plus a pole at 0 of weight 1/zeta_i^2,
//   g(nu) = b - nu - (1/zeta_i^2) sum_{j != i} zeta_j^2 / (Delta_j (1 - nu Delta_j))
//           + (1/zeta_i^2) / nu,
// and lambda = d_i + 1/nu for its extreme eigenvalue nu (bisection or the accelerated solve).
// The eigenvector is v = [x; -1] / ||.||, x_j = zeta_j / ((d_j - sigma) - mu).
//
// Then, as for D + rho z z^T (Sec. 2): where K_nu of Eq. (K0) is large the other neighbouring
// pole (R1) or a non-pole shift sigma next to lambda (R2) is taken.  For sigma not a pole,
// with f(sigma) the Schur complement of D - sigma I,
//   (A - sigma I)^{-1} = diag(e, 0) + gamma u u^T,  e_j = 1/(d_j - sigma),
//   u = [zeta_j/(d_j - sigma); -1],  gamma = 1/f(sigma),
// a DPR1 matrix of order n + 1 with a pole at 0 of weight gamma (the arrowhead form of
// Eq. (gamma)); its extreme eigenvalue is 1/(lambda - sigma).  sigma = 0 recomputes an
// eigenvalue much closer to zero than to its neighbouring poles.
//
// The matrix is first normalised by an exact power of two, A' = 2^-a A with
// max(|d_j|, |zeta_j|, |alpha|) = m 2^a, m in [1/2, 1) (k_arrow_norm; the kernels then work on
// the copies d', z', alpha'), and lambda, sigma, mu are scaled back; pairs that need values
// outside the binary64 range are reported as DPR1_ERR_RANGE.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../../include/dpr1.h"
#include "dpr1_device.cuh"
#include "dpr1_internal.cuh"
#include "dpr1_solve.cuh"

namespace dpr1 {

static size_t a256a(size_t x) { return (x + 255) & ~(size_t)255; }

struct ArrowWs {
  unsigned* status;              // word 0: status; words 8..: counters (as the DPR1 header)
  unsigned* counters;
  unsigned long long* queue;     // work counter of the solve kernel
  double* zz;                    // zeta_j^2 = zz + zl exactly
  double* zl;
  double* sig;                   // shift of eigenvalue k (a pole, or sigma of R2)
  double* mu;
  int* shift;                    // pole index, -1 for a non-pole shift
  int* list;                     // eigenvalues flagged by K_nu
  double* fixinfo;               // per flagged slot: K_nu, K_nu at the other pole, distance ratio
  long long* dq;                 // for the shift tests, in fixinfo's bytes before it is filled (as Ws::dq)
  float* zf;
  int* zlist;                    // near-zero candidates
  double* lamz;                  // lambda recomputed from A^{-1} (NaN: not recomputed)
  double* ds;                    // d' = 2^-a d and z' = 2^-a z (normalised copies)
  double* zs;
  double* scal;                  // [0]: alpha' = 2^-a alpha; [1]: a (as a double)
  // elements of the inverse for the solves and their binary32 copies, laid out as Ws::terms
  double* terms;
  int64_t term_n;
  int64_t term_slots;
  // the eigenvector rows the solve kernel's tail writes, as Ws::vrow and Ws::vstate (nullptr: the
  // vectors kernel writes every row)
  double* vrow;
  unsigned* vstate;
};

static size_t arrow_layout(int64_t n, ArrowWs* w, char* base) {
  size_t nn = (size_t)(n > 0 ? n : 1) + 1;
  size_t off = 0;
  size_t o_h = off; off += 256;
  size_t o_zz = off; off += a256a(8 * nn);
  size_t o_zl = off; off += a256a(8 * nn);
  size_t o_s = off; off += a256a(8 * nn);
  size_t o_m = off; off += a256a(8 * nn);
  size_t o_sh = off; off += a256a(4 * nn);
  size_t o_l = off; off += a256a(4 * nn);
  size_t o_fi = off; off += a256a(24 * nn);
  size_t o_zl2 = off; off += a256a(4 * nn);
  size_t o_lz = off; off += a256a(8 * nn);
  size_t o_ds = off; off += a256a(8 * nn);
  size_t o_zs = off; off += a256a(8 * nn);
  size_t o_sc = off; off += 256;
  if (w && base) {
    w->status = (unsigned*)(base + o_h);
    w->counters = (unsigned*)(base + o_h) + 8;
    w->queue = (unsigned long long*)((unsigned*)(base + o_h) + 24);
    w->zz = (double*)(base + o_zz);
    w->zl = (double*)(base + o_zl);
    w->sig = (double*)(base + o_s);
    w->mu = (double*)(base + o_m);
    w->shift = (int*)(base + o_sh);
    w->list = (int*)(base + o_l);
    w->fixinfo = (double*)(base + o_fi);
    w->dq = (long long*)(base + o_fi);
    w->zf = (float*)(base + o_fi + 8 * nn);
    w->zlist = (int*)(base + o_zl2);
    w->lamz = (double*)(base + o_lz);
    w->ds = (double*)(base + o_ds);
    w->zs = (double*)(base + o_zs);
    w->scal = (double*)(base + o_sc);
    w->terms = nullptr;
    w->term_n = 0;
    w->term_slots = 0;
    w->vrow = nullptr;
    w->vstate = nullptr;
  }
  return off;
}

constexpr unsigned ST_FATAL_A = ST_NONFINITE | ST_UNSORTED | ST_BADARG;
// the solve kernel's shift test from the binary32 pass where its bound decides the sign
constexpr bool kArrowShift32 = DPR1_SHIFT32 != 0;
// orders n above which the solve kernel's tail writes eigenvector rows
constexpr int64_t kArrowTailMinN = 2048;
constexpr unsigned AH_ZERO_POLE = 1u;   // header word 1: some d_j == 0 (no near-zero recompute)
// remedies kernel: block-wide lane groups, two blocks per SM (as for D + rho z z^T)
constexpr int AH_FIX_THREADS = 256;
constexpr int AH_FIX_BLOCKS_PER_SM = 2;

// Exact power-of-two normalisation (one block): a from max(|d_j|, |zeta_j|, |alpha|) = m 2^a,
// m in [1/2, 1); the whole matrix scales by 2^-a, so lambda = 2^a lambda' and the eigenvectors
// are unchanged.  In the normal range this changes no rounding.
__global__ void k_arrow_norm(int n, const double* __restrict__ d, const double* __restrict__ z, double alpha,
                             double* __restrict__ scal) {
  double m = fabs(alpha);
  for (int j = threadIdx.x; j < n; j += blockDim.x) m = fmax(m, fmax(fabs(d[j]), fabs(z[j])));
  m = group_max<256>(m, FULL);
  if (threadIdx.x == 0) {
    int a = 0;
    if (m > 0.0 && isfinite(m)) frexp(m, &a);
    scal[0] = scalbn(alpha, -a);
    scal[1] = (double)a;
  }
}

// input checks (finite, strictly decreasing d, no zero weight), the normalised copies and zeta'^2
__global__ void k_arrow_check(int n, const double* __restrict__ d, const double* __restrict__ z, double alpha,
                              ArrowWs w) {
  const int a = (int)w.scal[1];
  double* __restrict__ zz = w.zz;
  double* __restrict__ zl = w.zl;
  unsigned* __restrict__ status = w.status;
  unsigned bits = 0, zp = 0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const double dj = d[j], zj = scalbn(z[j], -a);
    w.ds[j] = scalbn(dj, -a);
    w.zs[j] = zj;
    if (!isfinite(dj) || !isfinite(zj)) bits |= ST_NONFINITE;
    if (dj == 0.0) zp = AH_ZERO_POLE;
    if (j + 1 < n) {
      if (dj < d[j + 1]) bits |= ST_UNSORTED;
      else if (dj == d[j + 1]) bits |= ST_BADARG;       // equal poles: reducible
    }
    if (zero_weight(zj)) bits |= ST_BADARG;               // zero weight: reducible
    const double zq = __dmul_rn(zj, zj);
    zz[j] = zq;
    zl[j] = __fma_rn(zj, zj, -zq);
    w.dq[j] = pole_int(w.ds[j]);
    w.zf[j] = weight_f32(zq);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && !isfinite(alpha)) bits |= ST_NONFINITE;
  bits = __reduce_or_sync(FULL, bits);
  zp = __reduce_or_sync(FULL, zp);
  if ((threadIdx.x & 31) == 0 && bits) atomicOr(status, bits);
  if ((threadIdx.x & 31) == 0 && zp) atomicOr(status + 1, zp);
}

// Extreme eigenvalue nu of (A - d_i I)^{-1} on the side of eigenvalue k (rightmost when
// i == k, leftmost when i == k - 1); [alo, ahi] an estimate of the bracket of |nu|.
// FIRST, check and *ill: as solve_pole.
template <int L, bool NI = false, bool FIRST = false>
__device__ PoleResult solve_pole_arrow(const double* __restrict__ d, const double* __restrict__ zl,
                                       const double* __restrict__ zz, int n, double alpha, int k, int i, double alo,
                                       double ahi, int cap, bool fast, int lane, unsigned gm,
                                       double* __restrict__ Ds = nullptr, double* __restrict__ us = nullptr,
                                       bool screen = false, bool check = false) {
  PoleResult r;
  r.screened = 0;
  r.screened_near = 0;
  r.screened_df = 0;
  r.inferred = 0;
  r.probes = 0;
  r.steps = 0;
  double sq;
  const double di = d[i];
  // the corner's pass also stores the elements of the inverse when the group has a buffer (and
  // their binary32 copies for the screen, after the two binary64 arrays: us = Ds + n)
  float* const F = (Ds && screen && !fast) ? (float*)(us + n) : nullptr;
  bool rng_ok = false;
  float qa = 0.0f;
  dd acc = dd_pole_sum<L, false, FIRST>(d, zz, zl, n, i, di, lane, gm, &sq, nullptr, Ds, us, F, &rng_ok, 0.0,
                                        FIRST ? nullptr : &qa);
  const bool scr_ok = rng_ok && F;
  dd B = dd_add(two_sum(di, -alpha), acc);
  const dd Zi = {zz[i], zl[i]};
  const double b = dd_to_double(dd_div(B, Zi));
  const double inv = 1.0 / zz[i];
  const double wn2 = sq / Zi.hi + inv;          // squared border: w_j (j != i) and 1/zeta_i
  const double wn = root_t<FIRST>(wn2);
  const double side = (i == k) ? 1.0 : -1.0;
  double floor, E;
  // the caller's [alo, ahi] rests on the shift test (or the 2 x 2 interlacing bounds) and is
  // checked first where it binds; the bounds below are rigorous up to rounding
  const double alo_in = alo, ahi_in = ahi;
  alo = 0.0;
  ahi = INFINITY;
  if (side > 0) {
    // largest pole of g: the nearest pole above d_i (or, for i = 0, the farthest below), or 0
    const double dmax = (i > 0) ? quot_t<FIRST>(1.0, d[i - 1] - di) : (n > 1 ? quot_t<FIRST>(1.0, d[n - 1] - di) : -INFINITY);
    const double pmax = fmax(dmax, 0.0);
    floor = pmax;
    E = pmax;
    alo = fmax(alo, b);
    ahi = fmin(ahi, fmax(b, pmax) + wn);
    if (b > pmax) ahi = fmin(ahi, b + quot_t<FIRST>(wn2, b - pmax));
    // smallest pole: the nearest delta_j below d_i (or the farthest above), or 0
    const double dmin = (i + 1 < n) ? quot_t<FIRST>(1.0, d[i + 1] - di) : (n > 1 ? quot_t<FIRST>(1.0, d[0] - di) : INFINITY);
    quad_bracket<FIRST>(b, fmin(dmin, 0.0), pmax, wn2, &alo, &ahi);
  } else {
    const double dmin = (i + 1 < n) ? quot_t<FIRST>(1.0, d[i + 1] - di) : (n > 1 ? quot_t<FIRST>(1.0, d[0] - di) : INFINITY);
    const double pmin = fmin(dmin, 0.0);
    floor = -pmin;
    E = -pmin;
    alo = fmax(alo, -b);
    ahi = fmin(ahi, -fmin(b, pmin) + wn);
    if (b < pmin) ahi = fmin(ahi, -b + quot_t<FIRST>(wn2, pmin - b));
    const double dmx = (i > 0) ? quot_t<FIRST>(1.0, d[i - 1] - di) : (n > 1 ? quot_t<FIRST>(1.0, d[n - 1] - di) : -INFINITY);
    quad_bracket<FIRST>(-b, -fmax(dmx, 0.0), -pmin, wn2, &alo, &ahi);
  }
  const bool eager_lo = alo_in > alo, eager_hi = ahi_in < ahi;
  alo = fmax(alo, alo_in) * (1.0 - 0x1p-48);
  ahi = fmin(ahi, ahi_in) * (1.0 + 0x1p-48);
  const double size = fabs(b) + inv * (double)qa;       // and inv / |nu| of the pole at 0
  bool ok;
  int steps = 0;
  double nu;
  // the finishing step (as in solve_pole, with the pole at 0)
  const double finish = !FIRST && rng_ok && inv < 0x1p100 ? kFinishCond : 0.0;
  const float cf = (float)inv;
  auto fin = [&](double v, double* Fv, double* s, double* mag) -> bool {
    double S;
    float q;
    if (!(fabs(v) >= 0x1p-60 && fabs(v) <= 0x1p60)) return false;
    if (!stored_sum_slope_x<NI, L>(Ds, us, n, v, cf, 1.0f, lane, gm, &S, &q)) return false;
    const double ex = inv / v;
    const dd bv = two_sum(b, -v);
    *Fv = side * __dadd_rn(__fma_rn(-S, inv, bv.hi), __dadd_rn(bv.lo, ex));
    *mag = fabs(b) + fabs(S * inv) + fabs(ex);
    *s = (double)q + ex / v;
    return isfinite(q);
  };
  r.ill = false;
  if (!FIRST && check && (!rng_ok || size + inv / alo > kIllCond * alo)) {
    double Fv, s = 0.0, m;
    r.ill = !rng_ok || !fin(side * ahi, &Fv, &s, &m) || size + inv / alo > kIllCond * alo * (1.0 + s);
    r.steps = rng_ok;
    if (r.ill) return r;
  }
  uint64_t blo, bhi;
  start_bracket(&floor, alo, ahi, &blo, &bhi);
  if (fast && finish > 0.0 && bhi - blo <= kFinishWidth &&
      finish_root(blo, bhi, side, E, 1.0, finish, fin, &steps, &nu)) {
    ok = true;
  } else if (fast) {
    const int tried = steps;
    // F(t) = side g(side t) = side b - t + Psi(t), Psi(t) = -side S / zeta_i^2 + (1/zeta_i^2) / t
    auto ev = [&](double t, bool want, double* psi, double* dpsi) {
      const double v = side * t;
      double dS = 0.0;
      const double S = want ? elem_sum_d<L>(Ds, us, d, zz, n, i, di, v, lane, gm, &dS)
                            : elem_sum<L>(Ds, us, d, zz, n, i, di, v, lane, gm);
      const double Sz = __dmul_rn(S, inv);
      const double ex = inv / t;
      *psi = -side * Sz + ex;
      *dpsi = -__dmul_rn(dS, inv) - ex / t;
      const double g = __dadd_rn(__dsub_rn(__dsub_rn(b, v), Sz), inv / v);
      return side > 0 ? g : -g;
    };
    nu = side * accel_solve(ev, floor, alo, ahi, E, side * b, 1.0, 1.0, cap, &ok, &steps);
    steps += tried;
  } else {
    auto phi = [&](double v) {
      const double S = elem_sum<L, false, NI>(Ds, us, d, zz, n, i, di, v, lane, gm);
      return __dadd_rn(__dsub_rn(__dsub_rn(b, v), __dmul_rn(S, inv)), inv / v);
    };
    // binary32 screen as in solve_pole; the extra pole's term fl(inv / v) is the same in both
    // evaluations, and the bound also covers the rounding of the intermediate difference X
    auto decide = [&](const Screened& c, double v, double Sz, double ex, double* g, double* tl) -> bool {
      const double X = __dsub_rn(__dsub_rn(b, v), Sz);
      const double G = __dadd_rn(X, ex);
      const double tol = __fma_rn(inv, (double)c.x, 1.01 * 0x1p-51 * fabs(X));
      if (!mag_greater(G, tol)) return false;
      if (!mag_greater(G, __dadd_rn(tol, tol))) r.screened_near++;
      *g = G;
      *tl = tol;
      return true;
    };
    // the binary32 screen, then the double-float screen (as in solve_pole)
    int f32_fail = 0;
    auto scr = [&](double v, double* g, double* tl, int mode, double* psi, double* dpsi) -> bool {
      if (!scr_ok) return false;
      Screened c;
      const double ex = inv / v;                    // phi's term, bit for bit
      double Sz = 0.0;
      bool ok = false;
      if (mode == 0 || (mode < 0 && f32_fail < kScreen32Tries)) {
        c = psi ? screen_sum_x<NI, L, true>(F, F + n, n, v, lane, gm) : screen_sum_x<NI, L, false>(F, F + n, n, v, lane, gm);
        Sz = __dmul_rn(c.S, inv);
        ok = decide(c, v, Sz, ex, g, tl);
        if (ok) {
          if (mode < 0) f32_fail = 0;
        } else {
          if (mode == 0) return false;
          f32_fail++;
        }
      }
      if (!ok) {
        if (mode == 1) f32_fail = kScreen32Tries;   // the probes have reached the binary32 window
        if (!kScreenDf) return false;
        c = psi ? screen_df_sum_x<NI, L, true>(F, n, v, lane, gm) : screen_df_sum_x<NI, L, false>(F, n, v, lane, gm);
        Sz = __dmul_rn(c.S, inv);
        if (!decide(c, v, Sz, ex, g, tl)) return false;
        r.screened_df++;
      }
      // Psi and Psi' on t = |nu| as the accelerated solve forms them (with the pole at 0)
      if (psi) {
        *psi = -side * Sz + fabs(ex);
        *dpsi = -__dmul_rn((double)c.slope, inv) - quot_approx(ex, v);
      }
      return true;
    };
    // g > 0 below the root for the rightmost eigenvalue, g < 0 for the leftmost
    nu = bisect(phi, side, floor, alo, ahi, side > 0, cap, &ok, &steps, eager_lo, eager_hi, scr, &r.screened,
                kPredict && scr_ok, E, side * b, &r.inferred, &r.probes, finish, 1.0,
                fin);
  }
  r.nu = nu;
  r.mu = 1.0 / nu;
  r.b = b;
  r.ok = ok;
  r.dd = true;
  r.steps += steps;
  return r;
}

// As solve_pole_first (the bracket of an exterior eigenvalue comes from the caller).
template <int L>
__device__ __noinline__ PoleResult solve_pole_arrow_first(const double* __restrict__ d, const double* __restrict__ zl,
                                                          const double* __restrict__ zz, int n, double alpha, int k,
                                                          int i, double alo, double ahi, int cap, bool fast, int lane,
                                                          unsigned gm, double* __restrict__ Ds,
                                                          double* __restrict__ us, bool screen) {
  if (k > 0 && k < n) alo = 1.0 / __dmul_rn(__dsub_rn(d[k - 1], d[k]), 0.5);
  return solve_pole_arrow<L, true, true>(d, zl, zz, n, alpha, k, i, alo, ahi, cap, fast, lane, gm, Ds, us, screen);
}

// One eigenvector row v = [x; -1] / ||.|| by a warp: x_j = zeta_j / ((d_j - sigma) - mu), ||[x; -1]||
// with a scaled fallback when the plain sum of squares overflows or a reciprocal leaves the fast
// range.  With vr the row is written (x_j stored as formed, then rescaled in place; the last
// component -c by lane 0).  Returns *nrm = ||[x; -1]|| scale and *scale.
__device__ __forceinline__ void arrow_row_values(const double* __restrict__ d, const double* __restrict__ z, int n,
                                                 double s, double m, double* __restrict__ vr, int lane,
                                                 double* nrm_out, double* scale_out) {
  double q = 0.0;
  bool bad = false;
  for (int j = lane; j < n; j += 32) {
    const double den = __dsub_rn(__dsub_rn(d[j], s), m);
    const double x = __dmul_rn(z[j], rcp_nr(den));
    bad |= !rcp_in_range(den);
    if (vr) vr[j] = x;
    q = __fma_rn(x, x, q);
  }
  q = group_sum<32>(q, FULL);
  q = __dadd_rn(q, 1.0);                        // the last component, -1
  bad = group_any<32>(bad, FULL);
  double scale = 1.0;
  bool rewrite = false;
  if (bad || !(q < 1e300)) {
    double mx = 1.0;
    for (int j = lane; j < n; j += 32) mx = fmax(mx, fabs(__dmul_rn(z[j], rcp(__dsub_rn(__dsub_rn(d[j], s), m)))));
    mx = group_max<32>(mx, FULL);
    scale = 1.0 / mx;
    q = 0.0;
    for (int j = lane; j < n; j += 32) {
      const double x = __dmul_rn(z[j], rcp(__dsub_rn(__dsub_rn(d[j], s), m))) * scale;
      q = __fma_rn(x, x, q);
    }
    q = group_sum<32>(q, FULL);
    q = __fma_rn(scale, scale, q);
    rewrite = true;
  }
  const double nrm = sqrt(q);
  const double c = scale / nrm;
  *nrm_out = nrm;
  *scale_out = scale;
  if (!vr) return;
  if (lane == 0) vr[n] = -c;
  if (!rewrite) {
    for (int j = lane; j < n; j += 32) vr[j] = __dmul_rn(vr[j], c);
  } else {
    for (int j = lane; j < n; j += 32) vr[j] = __dmul_rn(z[j], rcp(__dsub_rn(__dsub_rn(d[j], s), m))) * c;
  }
}

// A row written by the solve kernel's tail, out of line, and its record (pair, norm, scale).
__device__ __noinline__ void arrow_tail_row(const double* __restrict__ d, const double* __restrict__ z, int n,
                                            double s, double m, double* __restrict__ vr, int lane,
                                            double* __restrict__ rec) {
  double nrm, scale;
  arrow_row_values(d, z, n, s, m, vr, lane, &nrm, &scale);
  if (lane == 0) {
    rec[0] = s;
    rec[1] = m;
    rec[2] = nrm;
    rec[3] = scale;
  }
}

// One lane group per eigenvalue k = 0..n (persistent grid, work counter).  Once the counter is
// exhausted, with eigenvectors and the rows' records in the workspace, the groups (warps) sweep the
// rows once in order and write those of the eigenvalues solved so far (as k_solve's tail does);
// k_arrow_vectors writes the others and rewrites a row whose pair the remedies changed.
template <int L>
__global__ void __launch_bounds__(256, DPR1_SOLVE_MIN_BLOCKS) k_arrow_solve(int n, const double* __restrict__ d,
                                                     const double* __restrict__ z, ArrowWs w, int gpw, int cap,
                                                     bool fast, bool screen, double* __restrict__ Vt, int64_t ldv) {
  if (*w.status & ST_FATAL_A) return;
  const double alpha = w.scal[0];       // d, z and alpha are the normalised copies
  const int lane = threadIdx.x & (L - 1);
  const unsigned gm = group_mask<L>();
  const int leader = (threadIdx.x & 31) & ~(L - 1);
  const double* __restrict__ zz = w.zz;
  const int sub = (threadIdx.x & 31) / L;
  if (sub >= gpw) return;               // gpw lane groups of each warp work
  const int64_t grp = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * gpw + sub;
  double* const Dbuf = (w.terms && grp < w.term_slots && n <= w.term_n) ? w.terms + 4 * grp * w.term_n : nullptr;
  for (;;) {
    long long gl = 0;
    if (lane == 0) gl = (long long)atomicAdd(w.queue, 1ull);
    gl = __shfl_sync(gm, gl, leader, 32);
    if (gl > n) {
      if constexpr (kTailRows && L == 32) {
        if (!fast && w.vstate && Vt) {
          for (;;) {
            // lane 0 claims the next row, reads its pair after the acquire load and passes it on
            unsigned r = 0, st = 0;
            double sr = 0.0, mr = 0.0;
            if (lane == 0) {
              r = atomicAdd(&w.counters[C_TROW], 1u);
              if (r <= (unsigned)n) st = ld_acquire(w.vstate + r);
              if (st == 1u) {
                sr = w.sig[r];
                mr = w.mu[r];
              }
            }
            r = __shfl_sync(gm, r, 0, 32);
            st = __shfl_sync(gm, st, 0, 32);
            if (r > (unsigned)n) break;
            if (st != 1u) continue;
            sr = __shfl_sync(gm, sr, 0, 32);
            mr = __shfl_sync(gm, mr, 0, 32);
            arrow_tail_row(d, z, n, sr, mr, Vt + (int64_t)r * ldv, lane, w.vrow + 4 * (int64_t)r);
            if (lane == 0) {
              w.vstate[r] = 2u;
              atomicAdd(&w.counters[C_TAILROWS], 1u);
            }
          }
        }
      }
      break;
    }
    const int k = (int)gl;
    int i;
    bool shift32 = false;
    double alo = 0.0, ahi = INFINITY;
    if (k == 0 || k == n) {
      // exterior: the 2 x 2 principal matrix [d_i zeta_i; zeta_i alpha] bounds |mu| from
      // below (interlacing), Weyl with ||z|| bounds it from above
      i = (k == 0) ? 0 : n - 1;
      double s = 0.0;
      for (int j = lane; j < n; j += L) s = __dadd_rn(s, zz[j]);
      s = group_sum<L>(s, gm);
      const double h = (k == 0) ? 0.5 * (d[0] - alpha) : 0.5 * (d[n - 1] - alpha);
      const double rt = sqrt(h * h + zz[i]);
      const double mlo = (k == 0) ? (h >= 0.0 ? zz[i] / (h + rt) : rt - h) : (h >= 0.0 ? h + rt : zz[i] / (rt - h));
      const double gap = (k == 0) ? alpha - d[0] : d[n - 1] - alpha;
      alo = 1.0 / (fmax(gap, 0.0) + sqrt(s));
      ahi = 1.0 / mlo;
    } else {
      // shift test at the midpoint m = d_k + tau: F = f(m), f decreasing; the binary32 pass
      // decides where its bound settles the sign (the binary64 pass's sign), else the binary64
      // pass runs
      const double dk = d[k];
      const double tau = __dmul_rn(__dsub_rn(d[k - 1], dk), 0.5);
      const double c = __dsub_rn(__dsub_rn(alpha, dk), tau);
      double sp = 0.0, sn = 0.0, F = 0.0;
      const int sf = (kArrowShift32 && screen) ? shift_test_arrow_f32<L>(w.dq, w.zf, n, k, tau, c, lane, gm) : 0;
      shift32 = sf != 0;
      if (!shift32) {
        for (int j = lane; j < n; j += L) {
          const double t = __dmul_rn(zz[j], rcp_c(__dsub_rn(__dsub_rn(d[j], dk), tau)));
          if (j < k) sp = __dadd_rn(sp, t);
          else sn = __dadd_rn(sn, t);
        }
        sp = group_sum<L>(sp, gm);
        sn = group_sum<L>(sn, gm);
        F = c - (sp + sn);
      }
      alo = quot(1.0, tau);
      // the upper bracket end from the binary64 pass's partial sums is left out when the
      // binary32 pass may decide (both paths then start the bisection from the same bracket):
      //   mu in (0, tau]:   zeta_k^2 nu <= sum_{j<k} zeta_j^2/((d_j - d_k) - tau) + d_k - alpha + tau
      //   mu in [-tau, 0):  zeta_{k-1}^2 |nu| <= -sum_{j>=k} zeta_j^2/((d_j - d_k) - tau) + alpha - d_{k-1} + tau
      if (sf != 0 ? sf < 0 : F < 0.0) {
        i = k;
        if (!kArrowShift32) ahi = (sp + (dk - alpha) + tau) / zz[k];
      } else {
        i = k - 1;
        if (!kArrowShift32) ahi = (-sn + (alpha - d[k - 1]) + tau) / zz[k - 1];
      }
      if (!(ahi > alo)) ahi = INFINITY;
    }
    double* const us = Dbuf ? Dbuf + n : nullptr;
    PoleResult pr;
    pr.steps = 0;
    pr.ill = k == 0 || k == n || !Dbuf;   // as k_solve
    if (!pr.ill)
      pr = solve_pole_arrow<L, true>(d, w.zl, zz, n, alpha, k, i, alo, ahi, cap, fast, lane, gm, Dbuf, us, screen,
                                     true);
    if (pr.ill) {
      const int checked = pr.steps;
      pr = solve_pole_arrow_first<L>(d, w.zl, zz, n, alpha, k, i, alo, ahi, cap, fast, lane, gm, Dbuf, us, screen);
      pr.steps += checked;
    }
    if (lane == 0) {
      if (pr.screened) atomicAdd(&w.counters[C_SCREEN], (unsigned)pr.screened);
      if (pr.screened_near) atomicAdd(&w.counters[C_SCREEN_NEAR], (unsigned)pr.screened_near);
      if (pr.screened_df) atomicAdd(&w.counters[C_SCREEN_DF], (unsigned)pr.screened_df);
      if (pr.inferred) atomicAdd(&w.counters[C_INFER], (unsigned)pr.inferred);
      if (pr.probes) atomicAdd(&w.counters[C_PROBE], (unsigned)pr.probes);
      if (shift32) atomicAdd(&w.counters[C_SHIFT32], 1u);
      w.sig[k] = d[i];
      w.mu[k] = pr.mu;
      w.shift[k] = i;
      atomicAdd(&w.counters[C_EVAL_SOLVE], (unsigned)pr.steps);
      atomicAdd(&w.counters[C_SOLVED], 1u);
      if (!pr.ok) atomicOr(w.status, ST_NOT_CONVERGED);
      if (w.vstate) st_release(w.vstate + k, 1u);     // (sigma, mu) written: the row may be formed
    }
  }
}

// Non-pole shift sigma (R2, and sigma = 0 for the near-zero recompute): mu = 1/nu for the
// extreme eigenvalue nu of (A - sigma I)^{-1} = diag(e, 0) + gamma u u^T (see the top of the
// file), whose secular function is h(nu) = 1 + gamma (S(nu) - 1/nu), S(nu) = sum_j u_j^2/(e_j - nu)
// the shift sum.  f(sigma) = alpha - sigma - sum_j zeta_j^2/(d_j - sigma) is formed in
// double-double; f(sigma) = 0 gives mu = 0 (lambda = sigma).  above / below: the poles next to
// sigma (-1: none on that side).  The poles of h on |nu| are the e_j and 0, so the largest
// of them is max(e_above, 0) (gamma > 0, nu the rightmost) or max(-e_below, 0) (gamma < 0).
// With OFS the shift is sigma + sigma_lo in double the working precision (as solve_nonpole).
template <int L, bool OFS = false>
__device__ double solve_nonpole_arrow(const double* __restrict__ d, const double* __restrict__ zl,
                                      const double* __restrict__ zz, int n, double alpha, double sigma, int above,
                                      int below, int cap, bool fast, int lane, unsigned gm, bool* ok,
                                      int* steps_out, double* __restrict__ Ds = nullptr,
                                      double* __restrict__ us = nullptr, double sigma_lo = 0.0) {
  double un2, cub;
  bool rng_ok = false;
  // the double-double pass also stores the elements for the solve when the group has a buffer
  const dd acc = dd_pole_sum<L, OFS>(d, zz, zl, n, -1, sigma, lane, gm, &un2, &cub, Ds, us, nullptr, &rng_ok,
                                     sigma_lo);
  const dd f = dd_add(OFS ? shift_diff(alpha, sigma, sigma_lo) : two_sum(alpha, -sigma), {-acc.hi, -acc.lo});
  *ok = true;
  *steps_out = 0;
  if (f.hi == 0.0 && f.lo == 0.0) return 0.0;
  const double gamma = dd_to_double(dd_div({1.0, 0.0}, f));
  const double uu = un2 + 1.0;                  // ||u||^2, u_n = -1
  const double emax = above >= 0 ? 1.0 / elem_diff<OFS>(d[above], sigma, sigma_lo) : -INFINITY;
  const double emin = below >= 0 ? 1.0 / elem_diff<OFS>(d[below], sigma, sigma_lo) : INFINITY;
  // Rayleigh quotient of u (the pole at 0 adds nothing to u^T diag(e, 0) u): a lower bound of
  // the rightmost and an upper bound of the leftmost eigenvalue; Weyl bounds the other side
  const double rq = cub / uu + gamma * uu;
  double side, floor, alo, ahi;
  if (gamma > 0.0) {
    side = 1.0;
    floor = fmax(emax, 0.0);
    alo = fmax(floor, rq * (1.0 - 0x1p-48));
    ahi = floor + gamma * uu;
  } else {
    side = -1.0;
    floor = fmax(-emin, 0.0);
    alo = fmax(floor, -rq * (1.0 - 0x1p-48));
    ahi = floor - gamma * uu;
  }
  ahi *= (1.0 + 0x1p-48);
  int steps;
  double nu;
  // F(t) = -h(side t) = |gamma| (-1/|gamma| + Psi(t)), Psi(t) = -side S(side t) + 1/t; every
  // pole of Psi lies at or below floor, the model pole
  const double ag = fabs(gamma);
  const double finish = rng_ok && ag > 0x1p-60 && ag < 0x1p100 ? kFinishCond : 0.0;
  auto fin = [&](double v, double* Fv, double* s, double* mag) -> bool {
    double S;
    float q;
    const double t = fabs(v);
    if (!(t >= 0x1p-60 && t <= 0x1p60)) return false;
    if (!stored_sum_slope_x<false, L>(Ds, us, n, v, (float)ag, (float)t, lane, gm, &S, &q)) return false;
    *Fv = -__fma_rn(gamma, __dsub_rn(S, 1.0 / v), 1.0);
    *s = ((double)q + ag / t) / t;
    *mag = 1.0 + ag * (fabs(S) + 1.0 / t);
    return isfinite(q);
  };
  if (fast) {
    uint64_t lo, hi;
    steps = 0;
    start_bracket(&floor, alo, ahi, &lo, &hi);
    if (finish > 0.0 && hi - lo <= kFinishWidth && finish_root(lo, hi, side, floor, 0.0, finish, fin, &steps, &nu)) {
      *steps_out = steps;
      return 1.0 / nu;
    }
    const int tried = steps;
    auto ev = [&](double t, bool want, double* psi, double* dpsi) {
      const double v = side * t;
      double dS = 0.0;
      const double S = want ? elem_sum_d<L, OFS>(Ds, us, d, zz, n, -1, sigma, v, lane, gm, &dS, sigma_lo)
                            : elem_sum<L, OFS>(Ds, us, d, zz, n, -1, sigma, v, lane, gm, sigma_lo);
      const double it = 1.0 / t;
      *psi = -side * S + it;
      *dpsi = -dS - it * it;
      return -__fma_rn(gamma, __dsub_rn(S, 1.0 / v), 1.0);
    };
    nu = side * accel_solve(ev, floor, alo, ahi, floor, -1.0 / ag, 0.0, ag, cap, ok, &steps);
    steps += tried;
  } else {
    auto phi = [&](double v) {
      const double S = elem_sum<L, OFS>(Ds, us, d, zz, n, -1, sigma, v, lane, gm, sigma_lo);
      return __fma_rn(gamma, __dsub_rn(S, 1.0 / v), 1.0);
    };
    // h < 0 between the floor and the root in both cases
    nu = bisect(phi, side, floor, alo, ahi, false, cap, ok, &steps, false, false, NoScreen(), nullptr, false, floor,
                0.0, nullptr, nullptr, finish, 0.0, fin);
  }
  *steps_out = steps;
  return 1.0 / nu;
}

// |lambda_m - p| = |(sigma_m - p) + mu_m|
__device__ __forceinline__ double arrow_dist(const ArrowWs& w, int m, double p) {
  return fabs(__dadd_rn(__dsub_rn(w.sig[m], p), w.mu[m]));
}

// K_nu = ||(A - d_i I)^{-1}||_2 / |nu| (Eq. (K0)).  The eigenvalues next to pole d_i are
// lambda_i (above) and lambda_{i+1} (below), one of them lambda_k, and the norm is the
// reciprocal distance from d_i to the spectrum, so K_nu = max(1, |mu_k| / |lambda_m - d_i|) with
// lambda_m the other one.  For K_nu > T_Knu the eigenvalue goes to k_arrow_fix with the other
// neighbouring pole o of lambda_k (none for the exterior eigenvalues):
//   K'  = max(1, |lambda_k - d_o| / |lambda_m' - d_o|),  ratio = |lambda_k - d_o| / |lambda_k - d_i|.
__global__ void k_arrow_classify(int n, const double* __restrict__ d, ArrowWs w, double T_Knu) {
  if (*w.status & ST_FATAL_A) return;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= n; k += gridDim.x * blockDim.x) {
    const int i = w.shift[k];
    const double di = d[i], mu = w.mu[k];
    const double mk = fabs(mu);
    const int m = (i == k) ? k + 1 : k - 1;
    const double K = fmax(1.0, mk / arrow_dist(w, m, di));
    if (K > T_Knu) {
      const int o = (i == k) ? k - 1 : k;
      double K2 = INFINITY, ratio = INFINITY;
      if (o >= 0 && o < n) {
        const double dko = fabs(__dadd_rn(__dsub_rn(di, d[o]), mu));
        const int m2 = (o == k) ? k + 1 : k - 1;
        K2 = fmax(1.0, dko / arrow_dist(w, m2, d[o]));
        ratio = dko / mk;
      }
      const unsigned slot = atomicAdd(&w.counters[C_FIX_N], 1u);
      w.list[slot] = k;
      w.fixinfo[3 * (size_t)slot] = K;
      w.fixinfo[3 * (size_t)slot + 1] = K2;
      w.fixinfo[3 * (size_t)slot + 2] = ratio;
    }
  }
}

// After a non-pole shift: (d_p - sigma) - mu to a neighbouring pole p cancels by more than 16.
__device__ __forceinline__ bool ah_pole_difference_cancels(double dp, double s, double m) {
  const double t = __dsub_rn(__dsub_rn(dp, s), m);
  return 16.0 * fabs(t) < __dadd_rn(fabs(__dsub_rn(dp, s)), fabs(m));
}

// Remedies for the flagged eigenvalues, one lane group each (work counter):
//  (R1) solve at the other neighbouring pole o when K' < K, K' <= T_Knu and ratio <= T_Knu
//       (beyond that the eigenvector formula at d_o cancels);
//  (R2) otherwise sigma = fl(lambda) of the first pole solution, moved into the interlacing
//       interval of lambda_k (exterior ends from Weyl's bounds), and the non-pole solve,
//       repeated at the new lambda while sigma is not nearer to lambda_k than to the
//       interval's poles (at most 3 solves), as for D + rho z z^T; when no binary64 number lies
//       between lambda_k and a neighbouring pole, with the shift in double the working
//       precision (at most 3 more solves).
template <int L>
__global__ void __launch_bounds__(L > 256 ? L : 256) k_arrow_fix(int n, const double* __restrict__ d, ArrowWs w,
                                                                   double T_Knu, int cap, bool fast, bool screen) {
  if (*w.status & ST_FATAL_A) return;
  const double alpha = w.scal[0];
  const int nfix = (int)w.counters[C_FIX_N];
  const int lane = threadIdx.x & (L - 1);
  const unsigned gm = group_mask<L>();
  const int leader = (threadIdx.x & 31) & ~(L - 1);
  // the solve kernel has finished: its lane-group buffers are free for the remedies' solves
  const int64_t grp = (int64_t)blockIdx.x * (blockDim.x / L) + threadIdx.x / L;
  double* const Ds = (w.terms && grp < w.term_slots && n <= w.term_n) ? w.terms + 4 * grp * w.term_n : nullptr;
  double* const us = Ds ? Ds + n : nullptr;
  __shared__ int item;
  for (;;) {
    int t = 0;
    if constexpr (L > 32) {
      if (threadIdx.x == 0) item = (int)atomicAdd(&w.counters[C_FIX_Q], 1u);
      __syncthreads();
      t = item;
      __syncthreads();
    } else {
      if (lane == 0) t = (int)atomicAdd(&w.counters[C_FIX_Q], 1u);
      t = __shfl_sync(gm, t, leader, 32);
    }
    if (t >= nfix) break;
    const int k = w.list[t];
    const int i = w.shift[k];
    const double di = d[i], mu = w.mu[k];
    const double K = w.fixinfo[3 * (size_t)t];
    const double K2 = w.fixinfo[3 * (size_t)t + 1];
    const double ratio = w.fixinfo[3 * (size_t)t + 2];
    double new_sig = di, new_mu = mu;
    int new_shift = i;
    bool done = false;
    const int o = (i == k) ? k - 1 : k;
    // R1 only when it will be taken (as for D + rho z z^T)
    if (o >= 0 && o < n && K2 < K && K2 <= T_Knu && ratio <= T_Knu) {
      const PoleResult pr = solve_pole_arrow<L>(d, w.zl, w.zz, n, alpha, k, o, 0.0, INFINITY, cap, fast, lane, gm,
                                                Ds, us, screen);
      if (!pr.ok && lane == 0) atomicOr(w.status, ST_NOT_CONVERGED);
      if (lane == 0) atomicAdd(&w.counters[C_EVAL_FIX], (unsigned)pr.steps);
      if (lane == 0 && pr.screened) atomicAdd(&w.counters[C_SCREEN], (unsigned)pr.screened);
      if (lane == 0 && pr.screened_near) atomicAdd(&w.counters[C_SCREEN_NEAR], (unsigned)pr.screened_near);
      if (lane == 0 && pr.screened_df) atomicAdd(&w.counters[C_SCREEN_DF], (unsigned)pr.screened_df);
      if (lane == 0 && pr.inferred) atomicAdd(&w.counters[C_INFER], (unsigned)pr.inferred);
      if (lane == 0 && pr.probes) atomicAdd(&w.counters[C_PROBE], (unsigned)pr.probes);
      new_sig = d[o]; new_mu = pr.mu; new_shift = o; done = true;
    }
    if (!done) {
      // the interlacing interval of lambda_k; the exterior ends from Weyl's bounds,
      // lambda_0 <= max(d_0, alpha) + ||z||, lambda_n >= min(d_{n-1}, alpha) - ||z||
      const bool lo_pole = k < n, hi_pole = k > 0;
      double zn = 0.0;
      if (!lo_pole || !hi_pole) {
        double zs = 0.0;
        for (int j = lane; j < n; j += L) zs = __dadd_rn(zs, w.zz[j]);
        zn = sqrt(group_sum<L>(zs, gm));
      }
      const double lo = lo_pole ? d[k] : fmin(d[n - 1], alpha) - zn;
      const double hi = hi_pole ? d[k - 1] : fmax(d[0], alpha) + zn;
      double sg = __dadd_rn(di, mu);                    // the first solution's lambda
      bool solved = false;
      for (int round = 0; round < 3; round++) {
        if (lo_pole && !(sg > lo)) sg = dnext_up(lo);
        if (!lo_pole && !(sg >= lo)) sg = lo;
        if (hi_pole && sg >= hi) sg = dnext_down(hi);
        if (!hi_pole && sg > hi) sg = hi;
        if ((lo_pole && !(sg > lo)) || (hi_pole && !(sg < hi))) break;
        bool ok;
        int st2;
        const double m2 = solve_nonpole_arrow<L>(d, w.zl, w.zz, n, alpha, sg, k > 0 ? k - 1 : -1, k < n ? k : -1,
                                                 cap, fast, lane, gm, &ok, &st2, Ds, us);
        if (!ok && lane == 0) atomicOr(w.status, ST_NOT_CONVERGED);
        if (lane == 0) atomicAdd(&w.counters[C_EVAL_FIX], (unsigned)st2);
        new_sig = sg; new_mu = m2; new_shift = -1; solved = true;
        // repeat while sigma is not nearer to lambda_k than to the interval's poles
        double room = INFINITY;
        if (lo_pole) room = sg - lo;
        if (hi_pole) room = fmin(room, hi - sg);
        if (fabs(m2) < 0.5 * room) break;
        sg = __dadd_rn(sg, m2);
      }
      // no binary64 number between lambda_k and a neighbouring pole (the interval holds none, or
      // the result's difference to a pole cancels): the shift in double the working precision,
      // sigma = base + sgn tau with base the pole end nearer the lower end of the interval
      // (d_k; d_{n-1} for k = n, whose interval lies below it), tau in (0, g) between two poles
      // or up to the Weyl end; lambda - base is returned against the nearer pole
      if (!solved || (lo_pole && ah_pole_difference_cancels(lo, new_sig, new_mu)) ||
          (hi_pole && ah_pole_difference_cancels(hi, new_sig, new_mu))) {
        const double sgn = lo_pole ? 1.0 : -1.0;
        const double base = lo_pole ? lo : hi;
        const dd g = (lo_pole && hi_pole) ? two_sum(hi, -lo) : dd{__dsub_rn(hi, lo), 0.0};
        const double gw = __dadd_rn(g.hi, g.lo);
        const double mid = (lo_pole && hi_pole) ? 0.5 * gw : gw;
        const dd te = dd_add(two_sum(new_sig, -base), {new_mu, 0.0});
        double tau = sgn * __dadd_rn(te.hi, te.lo), m2 = 0.0;
        for (int round = 0; round < 3; round++) {
          if (!(tau > 0.0) || !(tau <= gw) || (lo_pole && hi_pole && !(tau < gw))) tau = mid;
          bool ok;
          int st2;
          m2 = solve_nonpole_arrow<L, true>(d, w.zl, w.zz, n, alpha, base, k > 0 ? k - 1 : -1, k < n ? k : -1, cap,
                                            fast, lane, gm, &ok, &st2, Ds, us, sgn * tau);
          if (!ok && lane == 0) atomicOr(w.status, ST_NOT_CONVERGED);
          if (lane == 0) atomicAdd(&w.counters[C_EVAL_FIX], (unsigned)st2);
          double room = tau;
          if (lo_pole && hi_pole) room = fmin(room, gw - tau);
          if (fabs(m2) < 0.5 * room) break;
          tau = (round == 0) ? mid : __fma_rn(sgn, m2, tau);
        }
        const dd lm = two_sum(sgn * tau, m2);             // lambda - base
        if (lo_pole && hi_pole && lm.hi > 0.5 * gw) {
          const dd up = dd_add(lm, {-g.hi, -g.lo});       // lambda - d_{k-1}
          new_sig = hi;
          new_mu = __dadd_rn(up.hi, up.lo);
        } else {
          new_sig = base;
          new_mu = __dadd_rn(lm.hi, lm.lo);
        }
        new_shift = -1;
        if (lane == 0) atomicAdd(&w.counters[C_R2DD], 1u);
      }
    }
    if (lane == 0) {
      w.sig[k] = new_sig;
      w.mu[k] = new_mu;
      w.shift[k] = new_shift;
      if (new_shift == -1) atomicAdd(&w.counters[C_R2], 1u);
      else if (new_shift != i) atomicAdd(&w.counters[C_R1], 1u);
    }
  }
}

// Eigenvalues much closer to zero than to their neighbouring poles,
// T_zero |lambda| < min(|lambda - d_k|, |lambda - d_{k-1}|) (the poles that exist), when no pole
// is zero: lambda = 1/nu, nu the extreme eigenvalue of A^{-1} (the non-pole solve at sigma = 0).
__global__ void k_arrow_zero_detect(int n, const double* __restrict__ d, ArrowWs w, double T_zero) {
  if (*w.status & ST_FATAL_A) return;
  const bool zero_pole = (w.status[1] & AH_ZERO_POLE) != 0;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= n; k += gridDim.x * blockDim.x) {
    w.lamz[k] = __longlong_as_double(0x7ff8000000000000ll);
    if (zero_pole) continue;
    const double sg = w.sig[k], m = w.mu[k];
    const double lam = __dadd_rn(sg, m);
    double m1 = INFINITY;
    if (k < n) m1 = fabs(__dadd_rn(__dsub_rn(sg, d[k]), m));
    if (k > 0) m1 = fmin(m1, fabs(__dadd_rn(__dsub_rn(sg, d[k - 1]), m)));
    if (T_zero * fabs(lam) < m1) {
      const unsigned slot = atomicAdd(&w.counters[C_ZERO_N], 1u);
      w.zlist[slot] = k;
    }
  }
}

__global__ void __launch_bounds__(256) k_arrow_zero_solve(int n, const double* __restrict__ d, ArrowWs w, int cap,
                                                          bool fast) {
  if (*w.status & ST_FATAL_A) return;
  const double alpha = w.scal[0];
  const int nz = (int)w.counters[C_ZERO_N];
  // a block-wide lane group per candidate, in one of the solve kernel's buffers where it has them (one
  // warp without them took about 0.5 ms of a 2.4 ms call at n = 2300)
  double* const Ds = (w.terms && blockIdx.x < w.term_slots && n <= w.term_n)
                         ? w.terms + 4 * (int64_t)blockIdx.x * w.term_n : nullptr;
  for (int t = blockIdx.x; t < nz; t += gridDim.x) {
    const int k = w.zlist[t];
    // the poles next to 0: the first negative pole and the one before it (no pole is zero)
    int lo = 0, hi = n;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (d[mid] > 0.0) lo = mid + 1;
      else hi = mid;
    }
    bool ok;
    int st;
    const double lam0 = solve_nonpole_arrow<256>(d, w.zl, w.zz, n, alpha, 0.0, lo - 1, lo < n ? lo : -1, cap, fast,
                                                 threadIdx.x, FULL, &ok, &st, Ds, Ds ? Ds + n : nullptr);
    if (threadIdx.x == 0) {
      w.lamz[k] = lam0;
      atomicAdd(&w.counters[C_EVAL_FIX], (unsigned)st);
      if (!ok) atomicOr(w.status, ST_NOT_CONVERGED);
    }
  }
}

// Rows v_k = [x; -1] / ||.|| (one warp per row), lambda, sigma, mu, ||[x; -1]||.  A row the solve
// kernel's tail wrote (arrow_row_values, the same arithmetic) is kept when its record holds the
// final (sigma, mu).
__global__ void __launch_bounds__(256) k_arrow_vectors(int n, const double* __restrict__ d,
                                                       const double* __restrict__ z, ArrowWs w,
                                                       double* __restrict__ lambda, double* __restrict__ Vt,
                                                       int64_t ldv, double* __restrict__ sigma,
                                                       double* __restrict__ mu, double* __restrict__ xnorm) {
  if (*w.status & ST_FATAL_A) return;
  const int lane = threadIdx.x & 31;
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = wid; k <= n; k += nw) {
    const double s = w.sig[k], m = w.mu[k];
    double* vr = Vt ? Vt + k * ldv : nullptr;
    double nrm, scale;
    bool kept = false;
    if (w.vstate && vr && w.vstate[k] == 2u) {
      const double* rec = w.vrow + 4 * k;
      if (__double_as_longlong(rec[0]) == __double_as_longlong(s) &&
          __double_as_longlong(rec[1]) == __double_as_longlong(m)) {
        nrm = rec[2];
        scale = rec[3];
        kept = true;
      }
    }
    if (!kept) {
      arrow_row_values(d, z, n, s, m, vr, lane, &nrm, &scale);
      if (vr && lane == 0) atomicAdd(&w.counters[C_VECROWS], 1u);
    }
    const double c = scale / nrm;
    if (lane == 0) {
      // outputs in the caller's units (lambda, sigma, mu times 2^a; x is scale-free)
      const int a = (int)w.scal[1];
      const double lz = w.lamz[k];
      const double lam = isnan(lz) ? __dadd_rn(s, m) : lz;
      const double xn = nrm / scale;
      lambda[k] = scalbn(lam, a);
      if (sigma) sigma[k] = scalbn(s, a);
      if (mu) mu[k] = scalbn(m, a);
      if (xnorm) xnorm[k] = xn;
      // outside the binary64 range of the normalised problem, or a cancelling pole difference
      // after a non-pole shift (as for D + rho z z^T)
      bool out = !(fabs(m) >= 0x1p-1022) || !isfinite(m) || !isfinite(lam) || !(xn > 0.0) || !isfinite(xn) ||
                 !isfinite(c);
      if (w.shift[k] < 0) out = out || (k < n && ah_pole_difference_cancels(d[k], s, m)) ||
                                (k > 0 && ah_pole_difference_cancels(d[k - 1], s, m));
      if (out) atomicOr(w.status, ST_RANGE);
    }
  }
}

// n = 0: the 1 x 1 matrix [alpha]
__global__ void k_arrow_one(double alpha, double* lambda, double* Vt, double* sigma, double* mu, double* xnorm) {
  lambda[0] = alpha;
  if (sigma) sigma[0] = alpha;
  if (mu) mu[0] = 0.0;
  if (xnorm) xnorm[0] = 1.0;
  if (Vt) Vt[0] = -1.0;
}

// lane groups of the solve kernel's default launch (as default_lanes for one problem D + rho z z^T)
static int arrow_lanes(int64_t n) { return n <= 96 ? 8 : (n <= 384 ? 16 : 32); }

static int64_t arrow_groups(int64_t n, int gpw, int warps, int bps) {
  const int groups_per_block = gpw * warps;
  int64_t want = (n + 1 + groups_per_block - 1) / groups_per_block;
  int64_t grid = (int64_t)sm_count() * bps;
  if (want < grid) grid = want > 0 ? want : 1;
  int64_t need = grid * groups_per_block;
  const int64_t fixg = (n + 1 < (int64_t)sm_count() * AH_FIX_BLOCKS_PER_SM) ? n + 1
                                                                           : (int64_t)sm_count() * AH_FIX_BLOCKS_PER_SM;
  return fixg > need ? fixg : need;
}

// bytes of the stored-element buffers for the default launch (8 warps per block,
// DPR1_SOLVE_MIN_BLOCKS blocks per SM)
// bytes of the records of the rows the solve kernel's tail writes (after the buffers, 256-byte
// aligned): 4 doubles and a state word per row, for n above kArrowTailMinN
static size_t arrow_tail_bytes(int64_t n) {
  if (!kTailRows || n <= kArrowTailMinN) return 0;
  return 256 + a256a(sizeof(double) * 4 * (size_t)(n + 1)) + a256a(sizeof(unsigned) * (size_t)(n + 1));
}

static size_t arrow_term_bytes(int64_t n) {
  if (n <= 0) return 0;
  const int64_t tn = (n + 31) & ~(int64_t)31;
  return (size_t)arrow_groups(n, 32 / arrow_lanes(n), 8, DPR1_SOLVE_MIN_BLOCKS) * TERM_BYTES * (size_t)tn +
         arrow_tail_bytes(n);
}

// tb: workspace bytes beyond the required part, for the solves' stored elements (one
// buffer of TERM_BYTES n bytes per lane group, for as many groups as the bytes allow; the remedies
// reuse them after the solve kernel)
template <int L>
static dpr1_status launch_arrow(int n, const double* d, const double* z, ArrowWs* w, const Options& o, char* tail,
                                size_t tb, double* Vt, int64_t ldv, cudaStream_t st) {
  // one lane group per warp by default, also where it is narrower (as run_table's gpw)
  const int gpw = o.lanes ? 32 / L : 1;
  // fewer lane groups than 8-warp blocks on every SM hold: blocks of fewer warps, one per SM
  int warps = o.warps;
  if (o.warps_auto && o.bps_auto) {
    const int64_t w_need = ((int64_t)n + 1 + (int64_t)gpw * sm_count() - 1) / ((int64_t)gpw * sm_count());
    // no more lane groups (a last block rounds up) than the default launch's, which have buffers
    const int64_t most = ((int64_t)n + 1 + 8 * gpw - 1) / (8 * gpw) * (8 * gpw);
    warps = w_need < 8 ? (int)w_need : 8;
    while (warps < 8 && ((int64_t)n + warps * gpw) / (warps * gpw) * (warps * gpw) > most) warps++;
  }
  const int groups_per_block = gpw * warps;
  int64_t want = ((int64_t)n + 1 + groups_per_block - 1) / groups_per_block;
  int grid = sm_count() * o.bps;
  if (want < grid) grid = (int)(want > 0 ? want : 1);
  if (tb > 0) {
    // a buffer for every group of the solve and the remedies kernels, or none (so the sums are
    // formed the same way whichever group takes an eigenvalue)
    const int64_t tn = ((int64_t)n + 31) & ~(int64_t)31;
    const int64_t slots = (int64_t)(tb / (TERM_BYTES * (size_t)tn));
    const int64_t need = arrow_groups(n, gpw, warps, o.bps);
    if (slots >= need) {
      w->terms = (double*)tail;
      w->term_n = tn;
      w->term_slots = need;
      // after the buffers, the records of the eigenvector rows the solve kernel's tail writes
      if (kTailRows && L == 32 && Vt && !o.fast && n > kArrowTailMinN) {
        const size_t at = a256a((size_t)need * TERM_BYTES * (size_t)tn);
        const size_t rec = a256a(sizeof(double) * 4 * (size_t)(n + 1));
        if (at + rec + a256a(sizeof(unsigned) * (size_t)(n + 1)) <= tb) {
          w->vrow = (double*)(tail + at);
          w->vstate = (unsigned*)(tail + at + rec);
          if (cudaMemsetAsync(w->vstate, 0, sizeof(unsigned) * (size_t)(n + 1), st) != cudaSuccess)
            return DPR1_ERR_CUDA;
        }
      }
    }
  }
  k_arrow_solve<L><<<grid, 32 * warps, 0, st>>>(n, d, z, *w, gpw, o.cap, o.fast, o.screen, Vt, ldv);
  return DPR1_OK;
}

}  // namespace dpr1

using namespace dpr1;

extern "C" {

size_t dpr1_arrow_workspace_size(int64_t n) {
  if (n < 0) return 0;
  return arrow_layout(n, nullptr, nullptr) + arrow_term_bytes(n);
}

dpr1_status dpr1_arrow_eig(int64_t n, const double* d, const double* z, double alpha, double* lambda, double* Vt,
                           int64_t ldv, double* sigma, double* mu, double* xnorm, void* workspace,
                           size_t workspace_bytes, const dpr1_options* opt, dpr1_stream_t stream) {
  if (n < 0 || n > (int64_t)0x3fffffff - 1) return DPR1_ERR_ARG;
  if (!lambda || (n > 0 && (!d || !z))) return DPR1_ERR_ARG;
  if (Vt && ldv < n + 1) return DPR1_ERR_ARG;
  // the stored-element buffers at the end of the workspace are optional
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < arrow_layout(n, nullptr, nullptr))
    return DPR1_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  ArrowWs w;
  const size_t base = arrow_layout(n, &w, (char*)workspace);
  char* const tail = (char*)workspace + base;
  const size_t tb = workspace_bytes - base;
  if (cudaMemsetAsync(w.status, 0, 256, st) != cudaSuccess) return DPR1_ERR_CUDA;
  if (n == 0) {
    if (!std::isfinite(alpha)) return DPR1_ERR_NONFINITE;
    k_arrow_one<<<1, 1, 0, st>>>(alpha, lambda, Vt, sigma, mu, xnorm);
    return cudaGetLastError() == cudaSuccess ? DPR1_OK : DPR1_ERR_CUDA;
  }
  const Options o = resolve(opt);
  const int sms = sm_count();
  int cg = (int)((n + 255) / 256);
  if (cg > sms * 8) cg = sms * 8;
  k_arrow_norm<<<1, 256, 0, st>>>((int)n, d, z, alpha, w.scal);
  k_arrow_check<<<cg, 256, 0, st>>>((int)n, d, z, alpha, w);
  // from here on the kernels work on the normalised copies d' = 2^-a d, z' = 2^-a z, alpha'
  const double* ds = w.ds;
  const double* zs = w.zs;
  const int L = o.lanes ? o.lanes : arrow_lanes(n);
  dpr1_status ls;
  if (L == 8) ls = launch_arrow<8>((int)n, ds, zs, &w, o, tail, tb, Vt, ldv, st);
  else if (L == 16) ls = launch_arrow<16>((int)n, ds, zs, &w, o, tail, tb, Vt, ldv, st);
  else ls = launch_arrow<32>((int)n, ds, zs, &w, o, tail, tb, Vt, ldv, st);
  if (ls != DPR1_OK) return ls;
  int kg = (int)((n + 1 + 255) / 256);
  if (kg > sms * 8) kg = sms * 8;
  k_arrow_classify<<<kg, 256, 0, st>>>((int)n, ds, w, o.T_Knu);
  // one block-wide group per flagged eigenvalue: they are few (a few percent on graded or
  // clustered spectra) and each solve spans all n poles
  const int fg = (int)(n + 1 < (int64_t)sms * AH_FIX_BLOCKS_PER_SM ? n + 1 : (int64_t)sms * AH_FIX_BLOCKS_PER_SM);
  k_arrow_fix<AH_FIX_THREADS><<<fg, AH_FIX_THREADS, 0, st>>>((int)n, ds, w, o.T_Knu, o.cap, o.fast, o.screen);
  k_arrow_zero_detect<<<kg, 256, 0, st>>>((int)n, ds, w, o.T_zero);
  k_arrow_zero_solve<<<2, 256, 0, st>>>((int)n, ds, w, o.cap, o.fast);
  int64_t vg = (n + 1 + 7) / 8;
  if (vg > sms * 16) vg = sms * 16;
  k_arrow_vectors<<<(int)vg, 256, 0, st>>>((int)n, ds, zs, w, lambda, Vt, ldv, sigma, mu, xnorm);
  return cudaGetLastError() == cudaSuccess ? DPR1_OK : DPR1_ERR_CUDA;
}

}  // extern "C"

// dpr1_backward.cu -- adjoint of the DPR1 eigen-decomposition (no counterpart in the
// paper; built from its Eq. (Pick) and Eq. (Aeigenvec)).
//
// For eigenpair k with lambda_k = sigma_k + mu_k the columns are recomputed, not stored:
//   s_j = d_j - lambda_k = (d_j - sigma_k) - mu_k,  x_j = zeta_j / s_j,  v = x / ||x||.
// The implicit derivative of f(lambda_k) = 1 + rho sum zeta_j^2 / (d_j - lambda_k) = 0 gives
//   dlambda/dd_j = v_j^2,  dlambda/dzeta_j = -2 x_j / ||x||^2,  dlambda/drho = 1/(rho^2 ||x||^2),
// and with vbar = dL/dv_k, c = v . vbar, g = vbar - v c (so gbar = g / ||x|| is dL/dx):
//   lambdabar = dL/dlambda_k + sum_j g_j v_j / s_j
//   dbar_j   += lambdabar v_j^2 - g_j v_j / s_j
//   zbar_j   += (g_j / s_j - 2 lambdabar v_j) / ||x||
//   rhobar   += lambdabar / (rho ||x||)^2
// Evaluation (as in the oracle's reading): p is the index of the largest |v_p|.  Next to a
// pole v is within ~1e-10 of e_p; then g_p and the two parts of dbar_p cancel at the scale
// 1/s_p, so with S2 = sum_{j != p} v_j^2 (= 1 - v_p^2) and P = sum_{j != p} v_j vbar_j:
//   c = v_p vbar_p + P,  g_p = vbar_p S2 - v_p P,
//   Lam = dL/dlambda_k + sum_{j != p} g_j v_j / s_j,  T_p = g_p v_p / s_p,  lambdabar = Lam + T_p,
//   dbar_p += Lam v_p^2 - T_p S2,   zbar_p += (g_p / s_p (S2 - v_p^2) - 2 Lam v_p) / ||x||.
// Work split: warp w of a set of NWB warps takes rows k = w, w + NWB, ... and keeps
// its own partial rows of dbar and zbar in the workspace (no atomics), and a final kernel
// sums the partials in warp order, so the result does not depend on scheduling.  Each warp
// also keeps the reciprocals 1/s_j of its current row, formed in the first pass and read back by the
// second (each lane reads what it wrote).
// Two passes over a row (bound by the binary64 pipe, so counted in its instructions per component):
// the first forms the reciprocal and the component (6) and, in units of x, every sum but the largest
// component's term (5): each lane holds its largest component so far out of its sums and adds the
// smaller of it and the new one, by integer comparison and selection; the lanes' held components
// other than p are added at the end.  The second forms the contributions (8).  19 in all, against 27
// in three passes (norm and p, sums, contributions), and one read of the row of dL/dV less.  Where x
// or a sum leaves a safe range, the sums are formed again in units of v, as the three passes did.
// The problem is normalised as in the forward (D' = 2^-a D, z' = 2^-b z, rho' = 2^(2b-a) rho,
// sigma' = 2^-a sigma, mu' = 2^-a mu, dL/dlambda' = 2^a dL/dlambda) and the gradients are
// scaled back (dL/dd = 2^-a dL/dd', dL/dz = 2^-b dL/dz', dL/drho = 2^(2b-a) dL/drho'): in the
// normal range this changes no rounding, and it keeps data of any magnitude in range.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../../include/dpr1.h"
#include "dpr1_device.cuh"
#include "dpr1_internal.cuh"

namespace dpr1 {

// Warps per block of the row kernel: 152 blocks, one per SM of a GB300 (numbers fixed by n and the
// workspace, so that the partial sums and their order do not depend on the device).  The kernel is
// latency-bound, and each warp costs a pair of partial rows that the last kernel adds, so the count
// grows with the order; backward in ms with 7 / 14 / 16 / 21 / 24 warps: n = 2048 0.295 / 0.31, 4096
// 1.02 / 0.92, 8192 4.21 / 3.33, 16384 (14 to 21) 13.0 / 12.6 / 13.5, 32768 (21, 24, 28) 51.6 / 49.5 /
// 49.5.  A workspace of wpb_least's size, which holds fewer partial rows, is accepted and runs as many.
static int wpb(int64_t n) { return n > 24576 ? 24 : (n > 10240 ? 16 : (n > 3072 ? 14 : 7)); }
static int wpb_least(int64_t n) { return n > 24576 ? 21 : (n > 8192 ? 14 : 7); }

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct BwdWs {
  unsigned* status;
  int* ex;      // status words 2, 3: the exponents a, b of the normalisation
  double* pd;   // [NWB][n]
  double* pz;   // [NWB][n]
  double* rb;   // [NWB][n] the reciprocals 1/s_j of each warp's current row
  double* pr;   // [NWB]
  double* ds;   // [n] d' = 2^-a d
  double* zs;   // [n] z' = 2^-b z
};

static size_t bwd_layout(int64_t n, int wp, BwdWs* w, char* base) {
  size_t nn = (size_t)(n > 0 ? n : 1);
  size_t off = 0;
  size_t o_st = off; off += 256;
  const size_t nw = (size_t)152 * wp;
  size_t o_pd = off; off += a256(sizeof(double) * nn * nw);
  size_t o_pz = off; off += a256(sizeof(double) * nn * nw);
  size_t o_rb = off; off += a256(sizeof(double) * nn * nw);
  size_t o_pr = off; off += a256(sizeof(double) * nw);
  size_t o_ds = off; off += a256(sizeof(double) * nn);
  size_t o_zs = off; off += a256(sizeof(double) * nn);
  if (w && base) {
    w->status = (unsigned*)(base + o_st);
    w->ex = (int*)(base + o_st) + 2;
    w->ds = (double*)(base + o_ds);
    w->zs = (double*)(base + o_zs);
    w->pd = (double*)(base + o_pd);
    w->pz = (double*)(base + o_pz);
    w->rb = (double*)(base + o_rb);
    w->pr = (double*)(base + o_pr);
  }
  return off;
}

// The exponents of the normalisation (one block): max|d_j| = m 2^a, max|z_j| = m' 2^b.
__global__ void __launch_bounds__(1024) k_bwd_norm(int n, const double* __restrict__ d, const double* __restrict__ z, BwdWs w) {
  double md = 0.0, mz = 0.0;
#pragma unroll 8
  for (int j = threadIdx.x; j < n; j += 1024) {
    md = fmax(md, fabs(d[j]));
    mz = fmax(mz, fabs(z[j]));
  }
  md = group_max<1024>(md, FULL);
  mz = group_max<1024>(mz, FULL);
  if (threadIdx.x == 0) {
    int a = 0, b = 0;
    if (md > 0.0 && isfinite(md)) frexp(md, &a);
    if (mz > 0.0 && isfinite(mz)) frexp(mz, &b);
    w.ex[0] = a;
    w.ex[1] = b;
  }
}

// the normalised copies d' and z'
__global__ void k_bwd_scale(int n, const double* __restrict__ d, const double* __restrict__ z, BwdWs w) {
  const int a = w.ex[0], b = w.ex[1];
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    w.ds[j] = scalbn(d[j], -a);
    w.zs[j] = scalbn(z[j], -b);
  }
}

// the bits of |x|: the order of magnitudes as integers (a NaN is largest)
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

template <int WPB>
__global__ void __launch_bounds__(32 * WPB, 1) k_bwd_rows(int n, double rho_in, const double* __restrict__ sig,
                                                  const double* __restrict__ mu, const double* __restrict__ gl,
                                                  const double* __restrict__ gV, int64_t ldg, BwdWs w) {
  const int lane = threadIdx.x & 31;
  constexpr int NWB = 152 * WPB;
  const int wid = (threadIdx.x >> 5) * 152 + blockIdx.x;   // the last, partial round spreads over the SMs
  const int ea = w.ex[0], eb = w.ex[1];
  const double* __restrict__ d = w.ds;
  const double* __restrict__ z = w.zs;
  const double rho = scalbn(rho_in, 2 * eb - ea);
  double* __restrict__ pd = w.pd + (size_t)wid * n;
  double* __restrict__ pz = w.pz + (size_t)wid * n;
  double* __restrict__ rb = w.rb + (size_t)wid * n;
  double prho = 0.0;
  unsigned bad = 0;
  bool first = true;
  for (int k = wid; k < n; k += NWB) {
    const double s = scalbn(sig[k], -ea), m = scalbn(mu[k], -ea);
    const double* __restrict__ grow = gV ? gV + (int64_t)k * ldg : nullptr;
    // pass 1: the index p of the largest component (the smallest index among equal ones) and, over
    // j != p in units of x: S2 = sum x_j^2, P = sum vbar_j x_j, A = sum vbar_j x_j / s_j,
    // Bs = sum x_j^2 / s_j
    double xm = 0.0, rm = 0.0, gm_ = 0.0;      // the lane's largest component so far, held out
    int p = n;
    double S2 = 0.0, P = 0.0, A = 0.0, Bs = 0.0;
#pragma unroll 2
    for (int j = lane; j < n; j += 32) {
      double r = rcp(__dsub_rn(__dsub_rn(d[j], s), m));
      double g = grow ? grow[j] : 0.0;
      rb[j] = r;
      double x = __dmul_rn(z[j], r);
      if (abs_bits(x) > abs_bits(xm)) {
        double t = x; x = xm; xm = t;
        t = r; r = rm; rm = t;
        t = g; g = gm_; gm_ = t;
        p = j;
      }
      const double xr = __dmul_rn(x, r);
      S2 = __fma_rn(x, x, S2);
      P = __fma_rn(x, g, P);
      A = __fma_rn(g, xr, A);
      Bs = __fma_rn(x, xr, Bs);
    }
    double mx = fabs(xm);
    const int own = p;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      double omx = __shfl_xor_sync(FULL, mx, o);
      int op = __shfl_xor_sync(FULL, p, o);
      if (omx > mx || (omx == mx && op < p)) { mx = omx; p = op; }
    }
    // one p and mx in all lanes also where a component is not a number (no order)
    mx = __shfl_sync(FULL, mx, 0);
    p = __shfl_sync(FULL, p, 0);
    if (own != p) {
      const double xr = __dmul_rn(xm, rm);
      S2 = __fma_rn(xm, xm, S2);
      P = __fma_rn(xm, gm_, P);
      A = __fma_rn(gm_, xr, A);
      Bs = __fma_rn(xm, xr, Bs);
    }
    S2 = group_sum<32>(S2, FULL);
    P = group_sum<32>(P, FULL);
    A = group_sum<32>(A, FULL);
    Bs = group_sum<32>(Bs, FULL);
    if (p >= n) p = 0;
    const double sp = __dsub_rn(__dsub_rn(d[p], s), m);
    const double rp = rcp(sp);
    const double xp = __dmul_rn(z[p], rp);
    const double gvp = grow ? grow[p] : 0.0;
    double cv, nrm;                            // v_j = x_j cv, cv = 1 / ||x||
    // in units of x, no further from underflow than 2^-120 of the cotangents; overflow shows in the sums
    if (mx > 0x1p-60 && mx < 1e100 && isfinite(S2) && isfinite(P) && isfinite(A) && isfinite(Bs)) {
      nrm = sqrt(__fma_rn(xp, xp, S2));
      cv = 1.0 / nrm;
      const double c2 = cv * cv;
      S2 *= c2;
      P *= cv;
      A *= cv;
      Bs *= c2;
    } else {
      // ||x|| scaled by the largest component where needed, and the sums in units of v
      double q = 0.0, scale = 1.0;
      for (int j = lane; j < n; j += 32) {
        const double x = __dmul_rn(z[j], rb[j]);
        q = __fma_rn(x, x, q);
      }
      q = group_sum<32>(q, FULL);
      if (!(q < 1e300) || !(mx > 1e-140)) {
        scale = 1.0 / mx;
        q = 0.0;
        for (int j = lane; j < n; j += 32) {
          const double x = __dmul_rn(z[j], rb[j]) * scale;
          q = __fma_rn(x, x, q);
        }
        q = group_sum<32>(q, FULL);
      }
      nrm = sqrt(q);
      cv = scale / nrm;
      S2 = 0.0; P = 0.0; A = 0.0; Bs = 0.0;
      for (int j = lane; j < n; j += 32) {
        if (j == p) continue;
        const double r = rb[j], g = grow ? grow[j] : 0.0;
        const double v = __dmul_rn(z[j], r) * cv;
        const double vr = __dmul_rn(v, r);
        S2 = __fma_rn(v, v, S2);
        P = __fma_rn(v, g, P);
        A = __fma_rn(g, vr, A);
        Bs = __fma_rn(v, vr, Bs);
      }
      S2 = group_sum<32>(S2, FULL);
      P = group_sum<32>(P, FULL);
      A = group_sum<32>(A, FULL);
      Bs = group_sum<32>(Bs, FULL);
    }
    const double inv = cv;                    // 1 / ||x||
    const double vp = xp * cv;
    const double c = grow ? __fma_rn(vp, gvp, P) : 0.0;
    const double gp = grow ? __fma_rn(gvp, S2, -vp * P) : 0.0;
    const double Lam = (gl ? scalbn(gl[k], ea) : 0.0) + (grow ? __fma_rn(-c, Bs, A) : 0.0);
    const double Tp = __dmul_rn(gp, vp) * rp;
    const double lb = Lam + Tp;
    // pass 2: contributions.  With a = lambdabar v_j and h = g_j / s_j:
    //   dbar_j = v_j (a - h),  zbar_j = (h - 2 a) / ||x||
    const double lb2 = -2.0 * lb;
#pragma unroll 2
    for (int j = lane; j < n; j += 32) {
      const double r = rb[j];
      const double v = __dmul_rn(__dmul_rn(z[j], r), cv);
      const double g = grow ? __fma_rn(-v, c, grow[j]) : 0.0;
      const double h = __dmul_rn(g, r);
      const double e = __fma_rn(lb, v, -h), f = __fma_rn(lb2, v, h);
      double db, zb;
      if (first) {
        db = __dmul_rn(v, e);
        zb = __dmul_rn(inv, f);
      } else {
        db = __fma_rn(v, e, pd[j]);
        zb = __fma_rn(inv, f, pz[j]);
      }
      if (j == p) {
        db = __fma_rn(Lam * vp, vp, -Tp * S2);
        zb = inv * __fma_rn(gp * rp, __fma_rn(-vp, vp, S2), -2.0 * Lam * vp);
        if (!first) { db += pd[j]; zb += pz[j]; }
      }
      pd[j] = db;
      pz[j] = zb;
    }
    first = false;
    double t = inv / rho;
    prho = __fma_rn(lb, t * t, prho);
    if (!isfinite(lb) || !isfinite(nrm)) bad = 1;
  }
  if (lane == 0) {
    w.pr[wid] = prho;
    if (bad) atomicOr(w.status, ST_NONFINITE);
  }
}

// grad_d[j] = sum_w pd[w][j] over the warps w < min(n, nwt), likewise grad_z and grad_rho, in a fixed
// order: a block takes 32 columns and BR slices of the warps, each thread a slice's rows in order, and
// the slices are added in order.  Bound by the latency of the reads where a thread takes all rows (319 us
// at n = 4096 with 1064 rows, 16 blocks); 32 slices give every SM reads in flight.
constexpr int BR = 32;
__global__ void __launch_bounds__(32 * BR) k_bwd_reduce(int n, int nwt, BwdWs w, double* __restrict__ gd,
                                                        double* __restrict__ gz, double* __restrict__ grho) {
  __shared__ double sa[BR][32], sb[BR][32];
  const int nw = n < nwt ? n : nwt;
  const int ea = w.ex[0], eb = w.ex[1];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  for (int j0 = blockIdx.x * 32; j0 < n; j0 += gridDim.x * 32) {
    const int j = j0 + lane;
    double a = 0.0, b = 0.0;
    if (j < n) {
#pragma unroll 4
      for (int t = sl; t < nw; t += BR) {
        a += w.pd[(size_t)t * n + j];
        b += w.pz[(size_t)t * n + j];
      }
    }
    sa[sl][lane] = a;
    sb[sl][lane] = b;
    __syncthreads();
    if (sl < 2 && j < n) {
      double t = 0.0;
      for (int q = 0; q < BR; q++) t += sl == 0 ? sa[q][lane] : sb[q][lane];
      if (sl == 0) gd[j] = scalbn(t, -ea);
      else gz[j] = scalbn(t, -eb);
    }
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    double r = 0.0;
    for (int t = lane; t < nw; t += 32) r += w.pr[t];
    r = group_sum<32>(r, FULL);
    if (lane == 0) *grho = scalbn(r, 2 * eb - ea);
  }
}

}  // namespace dpr1

using namespace dpr1;

extern "C" {

size_t dpr1_backward_workspace_size(int64_t n) {
  if (n < 0) return 0;
  return bwd_layout(n, wpb(n), nullptr, nullptr);
}

dpr1_status dpr1_eig_backward(int64_t n, const double* d, const double* z, double rho, const double* sigma,
                              const double* mu, const double* grad_lambda, const double* grad_Vt, int64_t ldg,
                              double* grad_d, double* grad_z, double* grad_rho, void* workspace,
                              size_t workspace_bytes, const dpr1_options* opt, dpr1_stream_t stream) {
  (void)opt;
  if (n < 0 || n > (int64_t)0x3fffffff) return DPR1_ERR_ARG;
  if (!std::isfinite(rho) || !(rho > 0.0)) return DPR1_ERR_RHO;
  if (n == 0) return DPR1_OK;
  if (!d || !z || !sigma || !mu || !grad_d || !grad_z || !grad_rho) return DPR1_ERR_ARG;
  if (grad_Vt && ldg < n) return DPR1_ERR_ARG;
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < bwd_layout(n, wpb_least(n), nullptr, nullptr))
    return DPR1_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  BwdWs w;
  const int wp = workspace_bytes >= bwd_layout(n, wpb(n), nullptr, nullptr) ? wpb(n) : wpb_least(n);
  bwd_layout(n, wp, &w, (char*)workspace);
  if (cudaMemsetAsync(w.status, 0, 256, st) != cudaSuccess) return DPR1_ERR_CUDA;
  int g = (int)((n + 255) / 256);
  if (g > 4 * sm_count()) g = 4 * sm_count();
  k_bwd_norm<<<1, 1024, 0, st>>>((int)n, d, z, w);
  k_bwd_scale<<<g, 256, 0, st>>>((int)n, d, z, w);
  const auto rows = wp == 24 ? k_bwd_rows<24> : wp == 21 ? k_bwd_rows<21> : wp == 16 ? k_bwd_rows<16>
                    : wp == 14 ? k_bwd_rows<14> : k_bwd_rows<7>;
  rows<<<152, 32 * wp, 0, st>>>((int)n, rho, sigma, mu, grad_lambda, grad_Vt, ldg, w);
  int rg = (int)((n + 31) / 32);
  if (rg > 8 * sm_count()) rg = 8 * sm_count();
  k_bwd_reduce<<<rg, 32 * BR, 0, st>>>((int)n, 152 * wp, w, grad_d, grad_z, grad_rho);
  return cudaGetLastError() == cudaSuccess ? DPR1_OK : DPR1_ERR_CUDA;
}

}  // extern "C"

// Vector kernels of the outer float64 PCG recurrence (Section 6: CG
// preconditioned by one V-cycle), the precision boundary, permutations and
// the fused ionic update + right-hand side of the time step (Section 3.1).
// Dot products are reduced deterministically: a fixed grid writes one partial
// per block; they are summed in one order, by the last block to finish (residual
// norms) or by every block of the kernel that uses the sum (no ticket per block and
// no wait for a last block).
#pragma once
#include "../../include/aggmg.h"
#include "face_op.cuh"
#include "kernels.cuh"

namespace aggmg {

enum { TK_R = 0, TK_R0 = 1 };

// Loop control of the WHILE node, launched after the PCG set-up and at the end
// of every iteration: ends the loop once the solve is done, and after
// max_it + 2 iterations in any case. It is the only kernel that calls the
// device-side graph API, so every compute kernel stays visible to profilers.
static __global__ void k_loop_ctl(CGState* st) {
  if (st->done || st->guard >= st->max_it + 2) {
    st->done = 1;
    if (st->use_cond) cudaGraphSetConditional((cudaGraphConditionalHandle)st->cond, 0u);
  }
  st->rho = st->rz;
  st->guard += 1;
}

// Reset of the per-solve fields (and of the coarse-level kernel's grid
// barrier, if any); the options (rtol, atol, max_it, flexible, cond,
// use_cond) are written by the host before the launch.
static __global__ void k_cg_reset(CGState* st, GridBar* bar) {
  if (bar) {
    bar->count = 0u;
    bar->err = 0;
  }
  st->guard = 0;
  st->iter = 0;
  st->done = 0;
  st->status = 0;
  st->rho = st->alpha = st->beta = st->pq = st->rr = st->r0 = 0.0;
  st->rz = 0.0;
}

// Start of a solve: reset (with the coarse-level kernel's grid barrier, if
// any) and select the WHILE node that this launch ends.
static __global__ void k_cg_begin(CGState* st, unsigned long long cond, int use_cond, GridBar* bar) {
  if (bar) {
    bar->count = 0u;
    bar->err = 0;
  }
  st->iter = 0;
  st->done = 0;
  st->status = 0;
  st->rho = st->alpha = st->beta = st->pq = st->rr = st->r0 = 0.0;
  st->rz = 0.0;
  st->guard = 0;
  st->cond = cond;
  st->use_cond = use_cond;
}

static __global__ void k_set_opts(CGState* st, double rtol, double atol, int max_it, int flexible) {
  st->rtol = rtol;
  st->atol = atol;
  st->max_it = max_it;
  st->flexible = flexible;
}

static __global__ void k_noop() {}

// ||r0||, tolerance, early exit when already converged
static __global__ void __launch_bounds__(RED_NT) k_r0(const double* __restrict__ r, int64_t n, double* partials, CGState* st) {
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * RED_NT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RED_NT)
    s += r[i] * r[i];
  if (partial_and_last<RED_NT>(s, partials, &st->ticket[TK_R0])) {
    double rr = sum_partials<RED_NT>(partials, gridDim.x);
    if (threadIdx.x == 0) {
      st->ticket[TK_R0] = 0;
      st->rr = rr;
      st->r0 = sqrt(rr);
      st->tol = fmax(st->rtol * st->r0, st->atol);
      if (!isfinite(st->r0)) {
        st->status = -6;
        st->done = 1;
      } else if (st->r0 <= st->tol || st->r0 == 0.0) {
        st->done = 1;
      }
    }
  }
}

// x += alpha p; r -= alpha q; ||r||; convergence test. Fused with the
// V-cycle's input cast (r32 = (float) r, when r32 is given) and, for the
// flexible variant, the (r_new, z_old) product of the Polak-Ribiere beta (z_old:
// the previous V-cycle's result, still in its buffer). alpha = rho / (p, q) from
// the float64 product's npq partials. Both sums use the fixed grid and block
// order of the other reductions; the partials of (r, z_old) go to the p update.
// HBM (56 B per entry) and the float64 pipe (4 FMAs per entry) bound it alike: 39 us
// on 512^2 Q2, where the bytes take 19 us and the FMAs 15; 608 blocks instead of 304
// took 45 us.
template <typename TZ>
static __global__ void __launch_bounds__(RED_NT) k_cg_update(double* __restrict__ x, double* __restrict__ r,
                                                      const double* __restrict__ p, const double* __restrict__ q,
                                                      float* __restrict__ r32, const TZ* __restrict__ zold, int64_t n,
                                                      const double* pq_partials, int npq, double* partials,
                                                      double* rz_partials, CGState* st) {
  if (st->done) return;
  const double pq = all_sum_partials<RED_NT>(pq_partials, npq);
  const double alpha = st->rho / pq;
  const bool flex = st->flexible != 0;
  using Z2 = typename std::conditional<std::is_same<TZ, float>::value, float2, double2>::type;
  double s = 0.0, sz = 0.0;
  // pairs of entries per 16-byte access (n is even: whole 32-unit slices),
  // a scalar tail otherwise
  const int64_t n2 = n >> 1;
#pragma unroll 2
  for (int64_t i = (int64_t)blockIdx.x * RED_NT + threadIdx.x; i < n2; i += (int64_t)gridDim.x * RED_NT) {
    double2 xv = reinterpret_cast<double2*>(x)[i];
    double2 rv = reinterpret_cast<double2*>(r)[i];
    const double2 pv = reinterpret_cast<const double2*>(p)[i];
    const double2 qv = reinterpret_cast<const double2*>(q)[i];
    xv.x += alpha * pv.x;
    xv.y += alpha * pv.y;
    rv.x = rv.x - alpha * qv.x;
    rv.y = rv.y - alpha * qv.y;
    reinterpret_cast<double2*>(x)[i] = xv;
    reinterpret_cast<double2*>(r)[i] = rv;
    s += rv.x * rv.x;
    s += rv.y * rv.y;
    if (flex) {
      const Z2 zv = reinterpret_cast<const Z2*>(zold)[i];
      sz += rv.x * to_double(zv.x);
      sz += rv.y * to_double(zv.y);
    }
    if (r32) reinterpret_cast<float2*>(r32)[i] = make_float2(to_float(rv.x), to_float(rv.y));
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
    const int64_t i = n - 1;
    x[i] += alpha * p[i];
    const double ri = r[i] - alpha * q[i];
    r[i] = ri;
    s += ri * ri;
    if (flex) sz += ri * (double)zold[i];
    if (r32) r32[i] = (float)ri;
  }
  if (flex) {
    const double bz = block_sum<RED_NT>(sz);
    if (threadIdx.x == 0) rz_partials[blockIdx.x] = bz;
  }
  if (partial_and_last<RED_NT>(s, partials, &st->ticket[TK_R])) {
    double rr = sum_partials<RED_NT>(partials, gridDim.x);
    if (threadIdx.x == 0) {
      st->ticket[TK_R] = 0;
      st->pq = pq;
      st->alpha = alpha;
      st->rr = rr;
      st->iter += 1;
      double rn = sqrt(rr);
      if (!isfinite(rn)) {
        st->status = -6;
        st->done = 1;
      } else if (rn <= st->tol) {
        st->done = 1;
      } else if (st->iter >= st->max_it) {
        st->status = -5;
        st->done = 1;
      }
    }
  }
}

// per-block partials of (r, z), z the V-cycle's result in its own precision
template <typename TZ>
static __global__ void __launch_bounds__(RED_NT) k_zdot(const TZ* __restrict__ z, const double* __restrict__ r, int64_t n,
                                                 double* partials, const CGState* st) {
  if (st->done) return;
  double s = 0.0;
  using Z2 = typename std::conditional<std::is_same<TZ, float>::value, float2, double2>::type;
  const int64_t n2 = n >> 1;
#pragma unroll 2
  for (int64_t i = (int64_t)blockIdx.x * RED_NT + threadIdx.x; i < n2; i += (int64_t)gridDim.x * RED_NT) {
    const Z2 zv = reinterpret_cast<const Z2*>(z)[i];
    const double2 rv = reinterpret_cast<const double2*>(r)[i];
    s += rv.x * to_double(zv.x);
    s += rv.y * to_double(zv.y);
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) s += r[n - 1] * (double)z[n - 1];
  const double b = block_sum<RED_NT>(s);
  if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// p = z + beta p (INIT: p = z), beta from the partials (cg_beta); rho follows in k_loop_ctl
template <typename TZ, bool INIT>
static __global__ void __launch_bounds__(RED_NT) k_pupd(const TZ* __restrict__ z, double* __restrict__ p, int64_t n,
                                                 const double* partials, int np, CGState* st) {
  if (st->done) return;
  const double beta = cg_beta<RED_NT, INIT>(partials, np, st);
  using Z2 = typename std::conditional<std::is_same<TZ, float>::value, float2, double2>::type;
  const int64_t n2 = n >> 1;
#pragma unroll 2
  for (int64_t i = (int64_t)blockIdx.x * RED_NT + threadIdx.x; i < n2; i += (int64_t)gridDim.x * RED_NT) {
    const Z2 zv = reinterpret_cast<const Z2*>(z)[i];
    double2 pv = make_double2(to_double(zv.x), to_double(zv.y));
    if (!INIT) {
      const double2 po = reinterpret_cast<const double2*>(p)[i];
      pv.x += beta * po.x;
      pv.y += beta * po.y;
    }
    reinterpret_cast<double2*>(p)[i] = pv;
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0)
    p[n - 1] = INIT ? (double)z[n - 1] : (double)z[n - 1] + beta * p[n - 1];
}

template <typename TO, typename TI>
static __global__ void k_cast(const TI* __restrict__ in, TO* __restrict__ out, int64_t n, const CGState* st) {
  if (st && st->done) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (TO)in[i];
}

// dst[i*B + r] = src[perm[i]*B + r]  (caller order -> internal order)
template <typename TO, typename TI>
static __global__ void k_gather_units(const TI* __restrict__ src, TO* __restrict__ dst, const int64_t* __restrict__ perm,
                               int64_t n, int B) {
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= n * B) return;
  const int64_t i = id / B;
  const int r = (int)(id % B);
  dst[id] = (TO)src[perm[i] * B + r];
}
// dst[perm[i]*B + r] = src[i*B + r]  (internal order -> caller order)
template <typename TO, typename TI>
static __global__ void k_scatter_units(const TI* __restrict__ src, TO* __restrict__ dst, const int64_t* __restrict__ perm,
                                int64_t n, int B) {
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= n * B) return;
  const int64_t i = id / B;
  const int r = (int)(id % B);
  dst[perm[i] * B + r] = (TO)src[id];
}

// ---------------------------------------------------------------- ionic models
struct IonicParams {
  int model;
  double k, a, eps, gamma, mu1, mu2;
  agg_bueno_orovio_params bo;
  // inverses of Bueno-Orovio time constants (hi: above the unit step that selects)
  struct {
    double a0_lo, a0_hi, tau1plus, tau2plus, tau2inf, a2_lo, a2_hi, taufi, o_lo, o_hi, tausi;
  } inv;
};
inline IonicParams make_ionic(int model, double k, double a, double eps, double gamma, double mu1, double mu2,
                              const agg_bueno_orovio_params& b) {
  IonicParams p{model, k, a, eps, gamma, mu1, mu2, b, {}};
  if (model == 2) {
    p.inv = {1.0 / b.tau1p,   1.0 / ((b.tau1pp - b.tau1p) + b.tau1p), 1.0 / b.tau1plus,
             1.0 / b.tau2plus, 1.0 / b.tau2inf,
             1.0 / b.tau3p,   1.0 / ((b.tau3pp - b.tau3p) + b.tau3p), 1.0 / b.taufi,
             1.0 / b.tauo_p,  1.0 / ((b.tauo_pp - b.tauo_p) + b.tauo_p), 1.0 / b.tausi};
  }
  return p;
}

// Gates per DoF: FitzHugh-Nagumo and Aliev-Panfilov 1, Bueno-Orovio 3; gate g
// of DoF i lives at w[g * stride + i].
constexpr int kMaxGates = 3;
__host__ __device__ inline int ionic_gates(int model) { return model == 2 ? 3 : 1; }

__device__ __forceinline__ double unit_step(double z, double z0) { return z >= z0 ? 1.0 : 0.0; }
// The smoothed step S = (1 + tanh(k (z - z0))) / 2 = 1 / (1 + exp(t)), t = -2 k (z - z0),
// and 1 / (tau + dtau S). Where exp(t) is so large that tau exp(t) might overflow (t
// >= 50, tested on the high word), S is exp(-t) to the last bit.
__device__ __forceinline__ double smooth_step(double z, double z0, double k) {
  return 1.0 / (1.0 + exp(-2.0 * k * (z - z0)));
}
__device__ __forceinline__ double smooth_rate(double z, double z0, double k, double tau, double dtau) {
  const double t = -2.0 * k * (z - z0);
  if (__double2hiint(t) >= 0x40490000) return 1.0 / (tau + dtau * exp(-t));
  const double e1 = 1.0 + exp(t);
  return e1 / (dtau + tau * e1);
}

// Bueno-Orovio (Section 2.3.2, Eq. BuenoOrovio). The float64 pipe bounds these
// (2 FMAs per SM and clock on GB300; a division is ~10 of them, a tanh ~50), so
// divisions by parameters are products with the inverses in IonicParams::inv,
// the smoothed steps cost one exponential each, and a term behind a unit step is
// evaluated on its side only. Gate update of 5.3M DoFs: 1,928 -> 745 us.
// The three gate rates:
__device__ __forceinline__ void bueno_orovio_rates(const IonicParams& q, double u, const double* w, double* H) {
  const agg_bueno_orovio_params& p = q.bo;
  const double hv1 = unit_step(u, p.V1), hv1m = unit_step(u, p.V1m);
  const double hv2 = unit_step(u, p.V2), hvo = unit_step(u, p.Vo);
  const double a0 = (1.0 - hv1) * (hv1m != 0.0 ? q.inv.a0_hi : q.inv.a0_lo);
  const double b0 = -hv1 * q.inv.tau1plus;
  const double w0inf = 1.0 - hv1m;
  double a1 = 0.0;                                    // behind 1 - H_V2
  if (hv2 == 0.0) a1 = smooth_rate(u, p.V2m, p.k2, p.tau2p, p.tau2pp - p.tau2p);
  const double b1 = -hv2 * q.inv.tau2plus;
  const double ut = u * q.inv.tau2inf;
  const double w1inf = hvo * (p.winf_star - 1.0 + ut) + 1.0 - ut;
  const double a2 = hv2 != 0.0 ? q.inv.a2_hi : q.inv.a2_lo;
  const double w2inf = smooth_step(u, p.V3, p.k3);
  H[0] = (b0 - a0) * w[0] + a0 * w0inf;
  H[1] = (b1 - a1) * w[1] + a1 * w1inf;
  H[2] = -a2 * w[2] + a2 * w2inf;
}
// and I_ion:
__device__ __forceinline__ double bueno_orovio_current(const IonicParams& q, double u, const double* w) {
  const agg_bueno_orovio_params& p = q.bo;
  const double hv1 = unit_step(u, p.V1), hv2 = unit_step(u, p.V2), hvo = unit_step(u, p.Vo);
  const double ifi = -hv1 * (u - p.V1) * (p.Vhat - u) * w[0] * q.inv.taufi;
  double iso = (1.0 - hv2) * (u - p.uo) * (hvo != 0.0 ? q.inv.o_hi : q.inv.o_lo);
  if (hv2 != 0.0) iso += smooth_rate(u, p.Vso, p.kso, p.tauso_p, p.tauso_pp - p.tauso_p);
  const double isi = -hv2 * w[1] * w[2] * q.inv.tausi;
  return ifi + iso + isi;
}

// gate rates H(u, w) and I_ion(u, w) (w, H: ionic_gates(model) values)
__device__ __forceinline__ void ionic_rates(const IonicParams& p, double u, const double* w, double* H) {
  if (p.model == 2) bueno_orovio_rates(p, u, w, H);
  else if (p.model == 0) H[0] = p.eps * (u - p.gamma * w[0]);
  else H[0] = (p.eps + p.mu1 * w[0] / (u + p.mu2)) * (-w[0] - p.k * u * (u - p.a - 1.0));
}
__device__ __forceinline__ double ionic_current(const IonicParams& p, double u, const double* w) {
  if (p.model == 2) return bueno_orovio_current(p, u, w);
  const double cub = p.k * u * (u - p.a) * (u - 1.0);
  return p.model == 0 ? cub + w[0] : cub + u * w[0];
}

// gate values of DoF i (stride between gates) into g[]
__device__ __forceinline__ void load_gates(const double* w, int64_t stride, int64_t i, int ng, double* g) {
#pragma unroll
  for (int k = 0; k < kMaxGates; ++k) g[k] = (k < ng) ? w[k * stride + i] : 0.0;
}

static __global__ void k_ionic_update(IonicParams prm, double dt, int64_t n, const double* __restrict__ u,
                               double* __restrict__ w) {
  const int ng = ionic_gates(prm.model);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double g[kMaxGates], H[kMaxGates];
    load_gates(w, n, i, ng, g);
    ionic_rates(prm, u[i], g, H);
#pragma unroll
    for (int k = 0; k < kMaxGates; ++k)
      if (k < ng) w[k * n + i] = g[k] + dt * H[k];
  }
}

// ---- element-wise kernels of a time step: one thread per (element, row), U
// whole elements per block; vectors are read coalesced, and a row's entries of an
// element's mass block (column by column, M[c * B + r]) too. With one thread per
// element the 64-DoF blocks left most of the GPU idle (k_ionic_rhs on 13,824 Q3
// hexahedra: 332 us; Bueno-Orovio on 24,576 Q2 hexahedra: 870 us, now ~170).
template <int B> struct ElemRows {
  static constexpr int U = (B <= 64) ? 128 / B : 1, NT = (U * B + 31) / 32 * 32;
};
// sum_c M[c B + r] t_c with the element's t in shared memory
template <int B>
__device__ __forceinline__ double elem_mv(const double* __restrict__ M, int r, const double* t) {
  double s = 0.0;
  constexpr int kUnroll = (B <= 27) ? B : 16;
#pragma unroll kUnroll
  for (int c = 0; c < B; ++c) s += __ldcs(M + c * B + r) * t[c];
  return s;
}

// Time step prologue (Section 3.1):
//   w <- w + dt H(u, w);  f = I_app(t_{n+1}) mask - chi I(u, w_new);
//   b_e = M_e (c u_e + f_e)   (ionic current interpolation)
template <int B>
static __global__ void __launch_bounds__(ElemRows<B>::NT)
    k_ionic_rhs(const double* __restrict__ Me, const double* __restrict__ u, double* __restrict__ w,
                const double* __restrict__ mask, double* __restrict__ b, IonicParams prm, double dt, double chi,
                double c, double iapp_value, int64_t iapp_steps, const int64_t* __restrict__ step, int64_t n,
                int64_t wstride) {
  constexpr int U = ElemRows<B>::U;
  __shared__ double sh[U * B];
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  const size_t o = (size_t)unit * B + r;
  if (active) {
    const double ia = (*step < iapp_steps) ? iapp_value : 0.0;
    const int ng = ionic_gates(prm.model);
    const double ur = u[o];
    double g[kMaxGates], H[kMaxGates];
    load_gates(w, wstride, o, ng, g);
    ionic_rates(prm, ur, g, H);
#pragma unroll
    for (int k = 0; k < kMaxGates; ++k)
      if (k < ng) {
        g[k] += dt * H[k];
        w[k * wstride + o] = g[k];
      }
    sh[threadIdx.x] = c * ur + ia * mask[o] - chi * ionic_current(prm, ur, g);
  }
  __syncthreads();
  if (active) b[o] = elem_mv<B>(Me + (size_t)unit * B * B, r, sh + slot * B);
}

// BDF2 history at the start (second-order derivative start), per element:
//   u^{-1} = u - dt u',  chi C_m u' = I_app - chi I(u, w) - M^{-1} A u,
//   w^{-1} = w - dt H(u, w),   with M^{-1} A u = M_e^{-1} (A0 u)_e - c u.
template <int B>
static __global__ void __launch_bounds__(ElemRows<B>::NT)
    k_bdf2_start(const double* __restrict__ Minv, const double* __restrict__ A0u, const double* __restrict__ u,
                 const double* __restrict__ w, const double* __restrict__ mask, double* __restrict__ up,
                 double* __restrict__ wp, IonicParams prm, double dt, double chi, double cm, double c, double ia,
                 int64_t n, int64_t wstride) {
  constexpr int U = ElemRows<B>::U;
  __shared__ double sh[U * B];
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  const size_t o = (size_t)unit * B + r;
  if (active) sh[threadIdx.x] = A0u[o];
  __syncthreads();
  if (!active) return;
  const double t = elem_mv<B>(Minv + (size_t)unit * B * B, r, sh + slot * B);
  const int ng = ionic_gates(prm.model);
  const double ur = u[o];
  double g[kMaxGates], H[kMaxGates];
  load_gates(w, wstride, o, ng, g);
  ionic_rates(prm, ur, g, H);
  const double f0 = ia * mask[o] - chi * ionic_current(prm, ur, g);
  const double udot = (f0 - (t - c * ur)) / (chi * cm);
  up[o] = ur - dt * udot;
#pragma unroll
  for (int k = 0; k < kMaxGates; ++k)
    if (k < ng) wp[k * wstride + o] = g[k] - dt * H[k];
}

// BDF2 step prologue (Eq. fully_discrete with extrapolation), per element:
//   U* = 2u - up, W* = 2w - wp, w_new = (4w - wp)/3 + (2dt/3) H(U*, W*),
//   f = I_app mask - chi I(U*, w_new), b_e = M_e (chi C_m (4u - up)/(2dt) + f);
//   then the history shifts: up <- u, wp <- w, w <- w_new.
template <int B>
static __global__ void __launch_bounds__(ElemRows<B>::NT)
    k_ionic_rhs_bdf2(const double* __restrict__ Me, const double* __restrict__ u, double* __restrict__ up,
                     double* __restrict__ w, double* __restrict__ wp, const double* __restrict__ mask,
                     double* __restrict__ b, IonicParams prm, double dt, double chi, double cm, double iapp_value,
                     int64_t iapp_steps, const int64_t* __restrict__ step, int64_t n, int64_t wstride) {
  constexpr int U = ElemRows<B>::U;
  __shared__ double sh[U * B];
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  const size_t o = (size_t)unit * B + r;
  if (active) {
    const double ia = (*step < iapp_steps) ? iapp_value : 0.0;
    const int ng = ionic_gates(prm.model);
    const double un = u[o], upr = up[o];
    const double us = 2.0 * un - upr;
    double wn[kMaxGates], wpr[kMaxGates], ws[kMaxGates], w1[kMaxGates], H[kMaxGates];
    load_gates(w, wstride, o, ng, wn);
    load_gates(wp, wstride, o, ng, wpr);
#pragma unroll
    for (int k = 0; k < kMaxGates; ++k) ws[k] = 2.0 * wn[k] - wpr[k];
    ionic_rates(prm, us, ws, H);
    up[o] = un;
#pragma unroll
    for (int k = 0; k < kMaxGates; ++k)
      if (k < ng) {
        w1[k] = (4.0 * wn[k] - wpr[k]) / 3.0 + (2.0 * dt / 3.0) * H[k];
        wp[k * wstride + o] = wn[k];
        w[k * wstride + o] = w1[k];
      } else {
        w1[k] = 0.0;
      }
    sh[threadIdx.x] = chi * cm / (2.0 * dt) * (4.0 * un - upr) + ia * mask[o] - chi * ionic_current(prm, us, w1);
  }
  __syncthreads();
  if (active) b[o] = elem_mv<B>(Me + (size_t)unit * B * B, r, sh + slot * B);
}

// Partial derivatives of the ionic model at one DoF (I_u, I_w, H_u, H_w).
__device__ __forceinline__ void ionic_jac(const IonicParams& p, double u, double w, double& Iu, double& Iw,
                                          double& Hu, double& Hw) {
  const double dcub = p.k * (3.0 * u * u - 2.0 * (p.a + 1.0) * u + p.a);
  if (p.model == 0) {
    Iu = dcub;
    Iw = 1.0;
    Hu = p.eps;
    Hw = -p.eps * p.gamma;
  } else {
    Iu = dcub + w;
    Iw = u;
    const double den = u + p.mu2;
    const double e = p.eps + p.mu1 * w / den;
    const double g = -w - p.k * u * (u - p.a - 1.0);
    const double e_u = -p.mu1 * w / (den * den), e_w = p.mu1 / den;
    const double g_u = -p.k * (2.0 * u - p.a - 1.0);
    Hu = e_u * g + e * g_u;
    Hw = e_w * g - e;
  }
}

// Reverse of one time step, pointwise part
// (discrete adjoint of the step; lambda = K^{-1} ubar is the input):
//   q = M_e lambda_e,  w~ = wbar - chi I_w(u_n, w_np1) q,
//   ubar_n = q (c - chi I_u(u_n, w_np1)) + dt H_u(u_n, w_n) w~,
//   wbar_n = w~ (1 + dt H_w(u_n, w_n)),   with w_np1 = w_n + dt H(u_n, w_n).
template <int B>
static __global__ void __launch_bounds__(ElemRows<B>::NT)
    k_adj_pointwise(const double* __restrict__ Me, const double* __restrict__ lam, const double* __restrict__ u_n,
                    const double* __restrict__ w_n, double* __restrict__ ubar, double* __restrict__ wbar,
                    IonicParams prm, double dt, double chi, double c, int64_t n) {
  constexpr int U = ElemRows<B>::U;
  __shared__ double sh[U * B];
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  const size_t o = (size_t)unit * B + r;
  if (active) sh[threadIdx.x] = lam[o];
  __syncthreads();
  if (!active) return;
  const double q = elem_mv<B>(Me + (size_t)unit * B * B, r, sh + slot * B);
  const double un = u_n[o], wn = w_n[o];
  double H[kMaxGates], Iu, Iw, Hu, Hw, Iu1, Iw1, Hu1, Hw1;
  const double wg[kMaxGates] = {wn, 0.0, 0.0};
  ionic_rates(prm, un, wg, H);                        // one-gate models only
  const double w1 = wn + dt * H[0];
  ionic_jac(prm, un, w1, Iu1, Iw1, Hu1, Hw1);
  ionic_jac(prm, un, wn, Iu, Iw, Hu, Hw);
  const double wt = wbar[o] - chi * Iw1 * q;
  ubar[o] = q * (c - chi * Iu1) + dt * Hu * wt;
  wbar[o] = wt * (1.0 + dt * Hw);
}

// Per-element log-conductivity gradient, accumulated in the caller's order:
//   grad[e] -= lam_e^T Ke u_e + sum_faces [lam_e; lam_n]^T Y_e,F [u_e; u_n]
// with Ke the volume form and Y_e,F the face terms built with D_e, of which
// only the trace-structured parts are stored (the row-major parts of Mesh::Yc,
// one after the other, per element and local face): ee on e's face rows, ee on
// face columns of the other rows, en on n's face columns, ne on n's face rows, nn.
// One thread per (element, DoF), U elements per block: the threads read B
// consecutive entries per step, hold a column each (the parts with NF columns:
// N rows per step) and sum over the rows, one FMA per entry; HBM bounds it
// (one thread per element walked 28,672 entries in sequence for Q3 hexahedra).
template <int B>
static __global__ void __launch_bounds__(ElemRows<B>::NT)
    k_grad_logD(FaceView<double, B> F, const double* __restrict__ Ke, const double* __restrict__ Yc,
                const double* __restrict__ lam, const double* __restrict__ u, const int64_t* __restrict__ perm,
                double* __restrict__ grad, int64_t n) {
  using FI = FaceIdx<FaceShape<B>::D, FaceShape<B>::N>;
  constexpr int N = FaceShape<B>::N, NF = FI::NF, NFACE = 2 * FaceShape<B>::D, U = ElemRows<B>::U;
  constexpr int S2 = (B - NF) * NF / B, S5 = NF * NF / B;     // steps of the parts with NF columns
  __shared__ double sl[U * B], su[U * B], sln[U * NFACE * NF], sun[U * NFACE * NF];
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  const int64_t f0 = unit / SL * NFACE * SL + unit % SL;      // (slice, face 0, lane)
  double* lu = sl + slot * B;
  double* uu = su + slot * B;
  double* ln = sln + slot * NFACE * NF;
  double* un = sun + slot * NFACE * NF;
  if (active) {
    lu[r] = lam[(size_t)unit * B + r];
    uu[r] = u[(size_t)unit * B + r];
    for (int k = r; k < NFACE * NF; k += B) {
      const int f = k / NF;
      const int nb = F.nbr[f0 + f * SL];
      if (nb < 0) continue;
      const size_t o = (size_t)nb * B + FI::face(F.code[f0 + f * SL], k % NF);
      ln[k] = lam[o];
      un[k] = u[o];
    }
  }
  __syncthreads();
  double g = 0.0;
  if (active) {
    const int q = r / NF, cf = r % NF;
    // sum over steps of M[step B + r] y(step)
    auto col = [&](const double* M, auto steps, auto y) {
      constexpr int kSteps = decltype(steps)::value;
      double s = 0.0;
#pragma unroll 8
      for (int i = 0; i < kSteps; ++i) s += __ldcs(M + i * B + r) * y(i);
      return s;
    };
    using std::integral_constant;
    g = col(Ke + (size_t)unit * B * B, integral_constant<int, B>{}, [&](int i) { return lu[i]; }) * uu[r];
#pragma unroll 1
    for (int f = 0; f < NFACE; ++f) {
      if (F.nbr[f0 + f * SL] < 0) continue;
      const double* M = Yc + ((size_t)unit * NFACE + f) * 4 * NF * B;
      const double* lnf = ln + f * NF;
      const double* unf = un + f * NF;
      g += col(M, integral_constant<int, NF>{}, [&](int i) { return lu[FI::face(f, i)]; }) * uu[r];
      M += NF * B;
      g += col(M, integral_constant<int, S2>{}, [&](int i) { return lu[FI::off(f, i * N + q)]; }) * uu[FI::face(f, cf)];
      M += (B - NF) * NF;
      g += col(M, integral_constant<int, NF>{}, [&](int i) { return lu[i * N + q]; }) * unf[cf];
      M += B * NF;
      g += col(M, integral_constant<int, NF>{}, [&](int i) { return lnf[i]; }) * uu[r];
      M += NF * B;
      g += col(M, integral_constant<int, S5>{}, [&](int i) { return lnf[i * N + q]; }) * unf[cf];
    }
  }
  __syncthreads();
  if (active) lu[r] = g;                              // summed in a fixed order
  __syncthreads();
  if (active && r < NF) {
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < N; ++a) s += lu[a * NF + r];
    uu[r] = s;
  }
  __syncthreads();
  if (active && r == 0) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < NF; ++j) s += uu[j];
    grad[perm[unit]] -= s;
  }
}

// end of a time step: record the iteration count, advance the clock
static __global__ void k_step_end(const CGState* st, int64_t* step, int* iters, int* slot, int capacity, int* status) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const int s = *slot;
    if (s < capacity) iters[s] = st->iter;
    if (st->status != 0 && *status == 0) *status = st->status;
    *slot = s + 1;
    *step = *step + 1;
  }
}

}  // namespace aggmg

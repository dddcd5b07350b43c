// Matrix-free GMRES on the device (Algorithm 1, Step 4): Arnoldi with
// classical Gram-Schmidt applied twice (CGS2: two block-parallel projections
// instead of j sequential ones), Givens rotations of the Hessenberg column on
// the device, restarts after `restart` steps.  Reductions are two-level and in
// a fixed order, so results are reproducible run to run.  The only host
// transfer per iteration is the residual estimate |g_{j+1}| (8 bytes).
#include <cmath>
#include <vector>

#include "kfbi_internal.cuh"

namespace kfbi {

kfbi_status apply_operator_impl(kfbi_problem* p, const double* x, double* y);

namespace {

constexpr int kDotThreads = 256;

// part[i * nchunk + c] = partial dot of V_i and w over chunk c
__global__ void k_dots(const double* __restrict__ V, int nb, int count,
                       const double* __restrict__ w, int nchunk, double* __restrict__ part) {
  const int i = blockIdx.y;
  const int c = blockIdx.x;
  const int per = (nb + nchunk - 1) / nchunk;
  const int b = c * per, e = min(nb, b + per);
  const double* v = V + (size_t)i * nb;
  double s = 0.0;
  for (int k = b + threadIdx.x; k < e; k += blockDim.x) s += v[k] * w[k];
  s = warp_sum(s);
  __shared__ double ws[kDotThreads / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = threadIdx.x < kDotThreads / 32 ? ws[threadIdx.x] : 0.0;
    t = warp_sum(t);
    if (threadIdx.x == 0) part[(size_t)i * nchunk + c] = t;
  }
}

// out[i] = (accumulate ? out[i] : 0) + sum_c part[i * nchunk + c], one block per i
__global__ void k_reduce(const double* __restrict__ part, int nchunk, double* __restrict__ out,
                         int accumulate) {
  const int i = blockIdx.x;
  double s = 0.0;
  for (int c = threadIdx.x; c < nchunk; c += blockDim.x) s += part[(size_t)i * nchunk + c];
  s = warp_sum(s);
  __shared__ double ws[kDotThreads / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = threadIdx.x < kDotThreads / 32 ? ws[threadIdx.x] : 0.0;
    t = warp_sum(t);
    if (threadIdx.x == 0) out[i] = accumulate ? out[i] + t : t;
  }
}

__global__ void k_scale(double* __restrict__ w, int nb, const double* __restrict__ s, int invert) {
  double f = invert ? 1.0 / s[0] : s[0];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nb; k += gridDim.x * blockDim.x)
    w[k] = w[k] * f;
}

__global__ void k_sub(const double* __restrict__ b, double* __restrict__ w, int nb) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nb; k += gridDim.x * blockDim.x)
    w[k] = b[k] - w[k];
}

__global__ void k_sqrt(double* s) { s[0] = sqrt(s[0]); }

__global__ void k_init_g(double* g, int m, const double* beta) {
  for (int i = threadIdx.x; i <= m; i += blockDim.x) g[i] = (i == 0) ? beta[0] : 0.0;
}

// upper-triangular solve H y = g (k x k)
__global__ void k_solve_y(const double* __restrict__ H, int ld, int k, const double* __restrict__ g,
                          double* __restrict__ y) {
  for (int i = k - 1; i >= 0; --i) {
    double s = g[i];
    for (int j = i + 1; j < k; ++j) s -= H[(size_t)j * ld + i] * y[j];
    y[i] = s / H[(size_t)i * ld + i];
  }
}

// x += sum_{i<k} y[i] V_i
__global__ void k_update_x(const double* __restrict__ V, int nb, int k, const double* __restrict__ y,
                           double* __restrict__ x) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nb; e += gridDim.x * blockDim.x) {
    double s = x[e];
    for (int i = 0; i < k; ++i) s += y[i] * V[(size_t)i * nb + e];
    x[e] = s;
  }
}

constexpr int kArnThreads = 1024;

// One Arnoldi step by one CTA (an instance of a batch): w = V_{j+1} holds A v_j on entry.
// CGS2 projections (each warp owns whole dot products), norm, normalisation
// and the Givens update of column j; res = |g_{j+1}|.
__device__ void arnoldi_step(double* __restrict__ V, int nb, int j, double* __restrict__ H, int ld,
                             double* __restrict__ cs, double* __restrict__ sn, double* __restrict__ g,
                             double* __restrict__ res, double* sm) {
  const int nw = kArnThreads / 32;
  double* part = sm;                       // (j+2) x nw
  double* h = part + (size_t)(j + 2) * nw; // j+2
  double* hacc = h + (j + 2);              // j+2
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* w = V + (size_t)(j + 1) * nb;
  for (int i = tid; i <= j + 1; i += kArnThreads) hacc[i] = 0.0;
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = warp; i <= j; i += nw) {
      const double* v = V + (size_t)i * nb;
      double s = 0.0;
      for (int k = lane; k < nb; k += 32) s += v[k] * w[k];
      s = warp_sum(s);
      if (lane == 0) {
        h[i] = s;
        hacc[i] += s;
      }
    }
    __syncthreads();
    for (int k = tid; k < nb; k += kArnThreads) {
      double s = w[k];
      for (int i = 0; i <= j; ++i) s -= h[i] * V[(size_t)i * nb + k];
      w[k] = s;
    }
    __syncthreads();
  }
  double s = 0.0;
  for (int k = tid; k < nb; k += kArnThreads) s += w[k] * w[k];
  s = warp_sum(s);
  if (lane == 0) part[warp] = s;
  __syncthreads();
  if (tid == 0) {
    double nn = 0.0;
    for (int q = 0; q < nw; ++q) nn += part[q];
    double hn = sqrt(nn);
    double* col = H + (size_t)j * ld;
    for (int i = 0; i <= j; ++i) col[i] = hacc[i];
    col[j + 1] = hn;
    for (int i = 0; i < j; ++i) {
      double t = cs[i] * col[i] + sn[i] * col[i + 1];
      col[i + 1] = -sn[i] * col[i] + cs[i] * col[i + 1];
      col[i] = t;
    }
    double rr = hypot(col[j], col[j + 1]);
    cs[j] = col[j] / rr;
    sn[j] = col[j + 1] / rr;
    col[j] = rr;
    col[j + 1] = 0.0;
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    res[0] = fabs(g[j + 1]);
    h[0] = hn;
  }
  __syncthreads();
  const double inv = 1.0 / h[0];
  for (int k = tid; k < nb; k += kArnThreads) w[k] *= inv;
}

}  // namespace

// ---- batched Arnoldi over instances (iteration counters on the device) -------


namespace {

__global__ void k_copy_in_batched(const ArnDesc* __restrict__ D, const int* __restrict__ jdev,
                                  const int* __restrict__ done) {
  const int k = blockIdx.y;
  if (done[k]) return;
  const ArnDesc& a = D[k];
  const double* v = a.V + (size_t)jdev[k] * a.nb;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < a.nb; e += gridDim.x * blockDim.x) a.x[e] = v[e];
}

__global__ void k_copy_out_batched(const ArnDesc* __restrict__ D, const int* __restrict__ jdev,
                                   const int* __restrict__ done) {
  const int k = blockIdx.y;
  if (done[k]) return;
  const ArnDesc& a = D[k];
  if (jdev[k] + 1 > a.m) return;
  double* v = a.V + (size_t)(jdev[k] + 1) * a.nb;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < a.nb; e += gridDim.x * blockDim.x) v[e] = a.y[e];
}

__global__ void __launch_bounds__(kArnThreads) k_arnoldi_batched(const ArnDesc* __restrict__ D,
                                                                 int* __restrict__ jdev,
                                                                 const int* __restrict__ done,
                                                                 double* __restrict__ res_out) {
  extern __shared__ double sm[];
  const int k = blockIdx.x;
  const ArnDesc& a = D[k];
  const int j = jdev[k];
  if (done[k] || j + 1 > a.m) {
    if (threadIdx.x == 0) res_out[k] = a.res[0];
    return;
  }
  arnoldi_step(a.V, a.nb, j, a.H, a.ld, a.cs, a.sn, a.g, a.res, sm);
  if (threadIdx.x == 0) {
    jdev[k] = j + 1;
    res_out[k] = a.res[0];
  }
}

}  // namespace

namespace {

// ---- one GMRES iteration on the device ----------------------------------------
// CGS2 across many CTAs with the step index j on the device: an Arnoldi step
// in one CTA is bound by that SM's FP64 rate (2 FMA/clk; at N_b = 29704 it took
// 0.60 ms an iteration), so each product V_i . w is cut into chunks of
// 2048 elements, a CTA each, and the update, which first adds its products'
// partial sums in a fixed order, runs on every SM (0.04 ms).
constexpr int kCgsThreads = 256;

// part[i nchunk + c] = V_i . w over chunk c, i <= j (CTAs beyond j exit); w is
// V_{j+1}, or the operator's output y in the first projection, which also takes
// over the step index: jdev[3], advanced by the step before, becomes jdev[0]
__global__ void __launch_bounds__(kCgsThreads) k_cgs_dots(const double* __restrict__ V, int nb,
                                                          int* __restrict__ jdev, int nchunk,
                                                          const double* __restrict__ y, double* __restrict__ part) {
  const int j = y ? jdev[3] : jdev[0];
  const int i = blockIdx.y, c = blockIdx.x;
  if (y && i == 0 && c == 0 && threadIdx.x == 0) jdev[0] = j;
  if (i > j) return;
  const double* v = V + (size_t)i * nb;
  const double* w = y ? y : V + (size_t)(j + 1) * nb;
  const int per = (nb + nchunk - 1) / nchunk;
  const int b = c * per, e = min(nb, b + per);
  double s = 0.0;
  for (int k = b + threadIdx.x; k < e; k += kCgsThreads) s += v[k] * w[k];
  s = warp_sum(s);
  __shared__ double ws[kCgsThreads / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kCgsThreads / 32; ++q) t += ws[q];
    part[(size_t)i * nchunk + c] = t;
  }
}

// h[i] = sum_c part[i nchunk + c]; V_{j+1} = w - sum_{i <= j} h[i] V_i, w = y or
// V_{j+1}; with npart: the CTA's sum of squares of the result
__global__ void __launch_bounds__(kCgsThreads) k_cgs_update(double* __restrict__ V, int nb,
                                                            const int* __restrict__ jdev,
                                                            const double* __restrict__ part, int nchunk,
                                                            const double* __restrict__ y, double* __restrict__ h,
                                                            double* __restrict__ npart) {
  const int j = jdev[0];
  __shared__ double hs[kMaxKrylov + 1];
  if (nchunk == 1) {
    for (int i = threadIdx.x; i <= j; i += kCgsThreads) hs[i] = part[i];
  } else {
    for (int i = threadIdx.x >> 5; i <= j; i += kCgsThreads / 32) {
      double s = 0.0;
      for (int c = threadIdx.x & 31; c < nchunk; c += 32) s += part[(size_t)i * nchunk + c];
      s = warp_sum(s);
      if ((threadIdx.x & 31) == 0) hs[i] = s;
    }
  }
  __syncthreads();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= j; i += kCgsThreads) h[i] = hs[i];
  double* w = V + (size_t)(j + 1) * nb;
  double acc = 0.0;
  for (int k = blockIdx.x * kCgsThreads + threadIdx.x; k < nb; k += gridDim.x * kCgsThreads) {
    double s = y ? y[k] : w[k];
    for (int i = 0; i <= j; ++i) s -= hs[i] * V[(size_t)i * nb + k];
    w[k] = s;
    acc += s * s;
  }
  if (!npart) return;
  acc = warp_sum(acc);
  __shared__ double ws[kCgsThreads / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kCgsThreads / 32; ++q) t += ws[q];
    npart[blockIdx.x] = t;
  }
}

// h_{j+1,j} = |V_{j+1}| (from the partials, in a fixed order, by every CTA);
// V_{j+1} /= h_{j+1,j}, also into x, the operator's input.  CTA 0 then adds the
// Hessenberg column h1 + h2, its Givens update, res = |g_{j+1}|, and advances the
// step index (jdev[3], which no CTA of this kernel reads).  With use_cond (the
// body of the device-driven loop): the loop continues while res > thr and j + 1
// < jdev[2], so it ends after at most jdev[2] iterations whatever the residual
// (NaN included).
__global__ void __launch_bounds__(kCgsThreads) k_cgs_finish(double* __restrict__ V, int nb, double* __restrict__ x,
                                                            double* __restrict__ H, int ld, double* __restrict__ cs,
                                                            double* __restrict__ sn, double* __restrict__ g,
                                                            double* __restrict__ res, const double* __restrict__ h1,
                                                            const double* __restrict__ h2,
                                                            const double* __restrict__ part, int npart,
                                                            int* __restrict__ jdev, cudaGraphConditionalHandle cond,
                                                            int use_cond, const double* __restrict__ thr) {
  __shared__ double ws[kCgsThreads / 32];
  const int j = jdev[0];
  double s = 0.0;
  for (int c = threadIdx.x; c < npart; c += kCgsThreads) s += part[c];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  double nn = 0.0;
  for (int q = 0; q < kCgsThreads / 32; ++q) nn += ws[q];
  const double hn = sqrt(nn);
  const double f = 1.0 / hn;
  double* w = V + (size_t)(j + 1) * nb;
  for (int k = blockIdx.x * kCgsThreads + threadIdx.x; k < nb; k += gridDim.x * kCgsThreads) {
    const double v = w[k] * f;
    w[k] = v;
    x[k] = v;
  }
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  double* col = H + (size_t)j * ld;
  double below = h1[0] + h2[0];        // the entry the next rotation turns
  for (int i = 0; i < j; ++i) {
    const double next = h1[i + 1] + h2[i + 1];
    col[i] = cs[i] * below + sn[i] * next;
    below = -sn[i] * below + cs[i] * next;
  }
  const double rr = hypot(below, hn);
  cs[j] = below / rr;
  sn[j] = hn / rr;
  col[j] = rr;
  col[j + 1] = 0.0;
  g[j + 1] = -sn[j] * g[j];
  g[j] = cs[j] * g[j];
  res[0] = fabs(g[j + 1]);
  jdev[3] = j + 1;
  if (use_cond) cudaGraphSetConditional(cond, (res[0] > thr[0] && j + 1 < jdev[2]) ? 1u : 0u);
}

// Inexact GMRES (relaxation of the operator's accuracy as the residual
// falls, after Simoncini & Szyld 2003 and Bouras & Fraysse 2005): before
// operator application j the refinement tolerance of the mixed box solves
// becomes max(base, omega rtol ||b|| / ||r_j||), with thr = rtol ||b|| and
// res = ||r_j|| the current estimate.  While GMRES runs, res > thr, so the
// tolerance stays below omega.
__global__ void k_relax_tol(const double* __restrict__ thr, const double* __restrict__ res, double omega,
                            double base, double* __restrict__ t1, double* __restrict__ t2) {
  double t = omega * thr[0] / res[0];
  if (!(t > base)) t = base;
  if (t1) *t1 = t;
  if (t2) *t2 = t;
}

}  // namespace

// The omega of the relaxed tolerance: cfg.relax, half of it for the mu-form, whose
// operator nearly annihilates the constants (by the contrast), so that what a solve
// leaves out reaches the solution larger by the contrast.  Error against that of
// unrelaxed solves / refinement steps, flowers, rtol 1e-8, by the margin of a first
// solve's stop (first_margin) and omega / cfg.relax, at cfg.relax 0.03, 0.05, 0.1:
//   grid, contrast     margin 10, whole                 margin 10 contrast, whole      the same, half
//   1024^2, 10         1.00/13  0.95/11  0.95/11        1.00/14  1.00/13  1.00/13      1.00/14  1.00/14  1.00/13
//   1024^2, 100        0.99/16  1.03/15  1.03/15        1.00/18  1.00/17  1.00/16      1.00/18  1.00/18  1.00/17
//   1024^2, 1000       1.02/17  1.02/17  1.34/14        1.00/21  0.99/20  1.23/17      1.00/22  1.00/21  0.99/20
//   512^2, 1000        0.87/17  0.87/17  0.95/14        1.00/21  1.00/21  1.03/18      1.00/23  1.00/22  1.00/21
//   1024^2, 10000      0.97/14  0.97/14  7.7e4/9        0.67/20  0.67/20  0.67/19      0.28/21  0.67/20  0.67/20
// The margin alone decides at 10000 (a margin of 10 fails); what is left at 1000 and
// 0.1 is the relaxation itself, which also never stopping at a first solve leaves
// (1.23/19).  The general kind shows neither: flower 512^2, margin 10, whole omega,
// contrast 4 1.00/24  1.00/22  1.00/20, contrast 25 0.93/28  0.93/28  0.95/26 (by
// the mu-form's rule 1.00/27..24 and 0.95/37..0.87/33; unrelaxed 48 and 84 steps).
double relax_omega(const kfbi_problem* p) {
  return p->cfg.kind == KFBI_INTERFACE_MU ? 0.5 * p->cfg.relax : p->cfg.relax;
}

// The relaxed refinement tolerance before an operator application inside
// GMRES (k_relax_tol), for the problem and its twin; nothing when relax = 0.
kfbi_status relax_box_tol(kfbi_problem* p) {
  if (!(p->cfg.relax > 0)) return KFBI_OK;
  Gmres& G = p->gm;
  double* t1 = box_tol_dev(p);
  double* t2 = p->twin ? box_tol_dev(p->twin) : nullptr;
  if (t1 || t2)
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_relax_tol<<<1, 1, 0, p->stream>>>(G.scal + 5, G.scal + 2, relax_omega(p),
                                                                       box_tol(p), t1, t2));
  return KFBI_OK;
}

namespace {

constexpr int kBatchThreads = 256;

// fixed-order sum of one value per thread over a CTA of kBatchThreads
__device__ double cta_sum(double v, double* ws) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int q = 0; q < kBatchThreads / 32; ++q) t += ws[q];
  __syncthreads();
  return t;
}

// Start of every instance's GMRES (a CTA per instance): ||b||; with a start x0
// (y = A x0 already in the instance's operator output) r0 = b - y is taken
// when ||r0|| < ||b|| (finite), else the zero start (the single solve's rule);
// V_0 = r/||r||, g = (||r||, 0, ...), threshold rtol ||b||; an instance whose
// start already meets it (or is not finite) is marked done.
// The refinement tolerance of instance k's box solves before its next
// iteration: relaxed as in the single solve (k_relax_tol), base when omega = 0.
__device__ __forceinline__ double relaxed_tol(double omega, double base, double thr, double res) {
  double t = omega * thr / res;
  return omega > 0.0 && t > base ? t : base;
}

__global__ void __launch_bounds__(kBatchThreads) k_batch_init(const ArnDesc* __restrict__ D,
                                                             const BatchInst* __restrict__ I, double rtol,
                                                             double* __restrict__ thr, double* __restrict__ bn,
                                                             int* __restrict__ done, int* __restrict__ jdev,
                                                             int* __restrict__ flags, double* __restrict__ res_out,
                                                             double omega, const double* __restrict__ base_tol,
                                                             double* __restrict__ tol) {
  __shared__ double ws[kBatchThreads / 32];
  __shared__ double sc[2];
  const int k = blockIdx.x;
  const ArnDesc& a = D[k];
  const BatchInst& in = I[k];
  const bool has_x0 = in.x0 != nullptr;
  double sb = 0.0, sr = 0.0;
  for (int e = threadIdx.x; e < a.nb; e += kBatchThreads) {
    const double bv = in.b[e];
    sb += bv * bv;
    if (has_x0) {
      const double r = bv - a.y[e];
      sr += r * r;
    }
  }
  const double bnorm = sqrt(cta_sum(sb, ws));
  const double rnorm = has_x0 ? sqrt(cta_sum(sr, ws)) : 0.0;
  const bool use = has_x0 && rnorm < bnorm;   // false for a NaN residual
  const double beta = use ? rnorm : bnorm;
  if (threadIdx.x == 0) {
    sc[0] = beta > 0.0 ? 1.0 / beta : 0.0;
    sc[1] = beta;
  }
  __syncthreads();
  const double f = sc[0];
  for (int e = threadIdx.x; e < a.nb; e += kBatchThreads)
    a.V[e] = (use ? in.b[e] - a.y[e] : in.b[e]) * f;
  for (int i = threadIdx.x; i <= a.m; i += kBatchThreads) a.g[i] = i == 0 ? beta : 0.0;
  if (threadIdx.x == 0) {
    const double t = rtol * bnorm;
    thr[k] = t;
    bn[k] = bnorm;
    flags[k] = has_x0 ? (use ? 1 : 2) : 0;
    done[k] = (beta > t) ? 0 : 1;
    jdev[k] = 0;
    a.res[0] = beta;
    res_out[k] = beta;
    if (tol) tol[k] = relaxed_tol(omega, base_tol[k], t, beta);
  }
}

// After each batched iteration: instances whose residual estimate reached
// their threshold (or is not finite) are marked done; ctl[0] counts the
// iterations, ctl[2] the instances still active; with use_cond the loop
// continues while some instance is active and ctl[0] < ctl[1].
__global__ void __launch_bounds__(kBatchThreads) k_batch_control(const double* __restrict__ res,
                                                                const double* __restrict__ thr,
                                                                int* __restrict__ done, int n,
                                                                int* __restrict__ ctl,
                                                                cudaGraphConditionalHandle cond, int use_cond,
                                                                double omega, const double* __restrict__ base_tol,
                                                                double* __restrict__ tol) {
  __shared__ int wa[kBatchThreads / 32];
  int active = 0;
  for (int k = threadIdx.x; k < n; k += kBatchThreads) {
    if (done[k]) continue;
    if (res[k] > thr[k]) {
      ++active;
      if (tol) tol[k] = relaxed_tol(omega, base_tol[k], thr[k], res[k]);
    } else {
      done[k] = 1;
    }
  }
  for (int o = 16; o > 0; o >>= 1) active += __shfl_xor_sync(0xffffffffu, active, o);
  if ((threadIdx.x & 31) == 0) wa[threadIdx.x >> 5] = active;
  __syncthreads();
  if (threadIdx.x != 0) return;
  int tot = 0;
  for (int q = 0; q < kBatchThreads / 32; ++q) tot += wa[q];
  ctl[0] += 1;
  ctl[2] = tot;
  if (use_cond) cudaGraphSetConditional(cond, (tot > 0 && ctl[0] < ctl[1]) ? 1u : 0u);
}

// x = (x0 if taken) + sum_{i < k} y_i V_i with H y = g (k x k upper
// triangular, k = the instance's iterations), a CTA per instance
__global__ void __launch_bounds__(kBatchThreads) k_batch_finish(const ArnDesc* __restrict__ D,
                                                               const BatchInst* __restrict__ I,
                                                               const int* __restrict__ jdev,
                                                               const int* __restrict__ flags) {
  __shared__ double y[kMaxKrylov];
  const int k = blockIdx.x;
  const ArnDesc& a = D[k];
  const BatchInst& in = I[k];
  const int kk = min(jdev[k], a.m);
  if (threadIdx.x == 0) {
    for (int i = kk - 1; i >= 0; --i) {
      double s = a.g[i];
      for (int j = i + 1; j < kk; ++j) s -= a.H[(size_t)j * a.ld + i] * y[j];
      y[i] = s / a.H[(size_t)i * a.ld + i];
    }
  }
  __syncthreads();
  const bool base = flags[k] == 1;
  for (int e = threadIdx.x; e < a.nb; e += kBatchThreads) {
    double s = base ? in.x0[e] : 0.0;
    for (int i = 0; i < kk; ++i) s += y[i] * a.V[(size_t)i * a.nb + e];
    in.out[e] = s;
  }
}

}  // namespace

kfbi_status batch_gmres_init(kfbi_problem* p0, const ArnDesc* d, const BatchInst* inst, int n, double rtol,
                             double* thr, double* bn, int* done, int* jdev, int* flags, double* res_out,
                             double omega, const double* base_tol, double* tol, cudaStream_t st) {
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_batch_init<<<n, kBatchThreads, 0, st>>>(d, inst, rtol, thr, bn, done, jdev,
                                                                            flags, res_out, omega, base_tol, tol));
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status batch_gmres_control(kfbi_problem* p0, const double* res, const double* thr, int* done, int n, int* ctl,
                                cudaGraphConditionalHandle cond, int use_cond, double omega,
                                const double* base_tol, double* tol, cudaStream_t st) {
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_batch_control<<<1, kBatchThreads, 0, st>>>(res, thr, done, n, ctl, cond,
                                                                               use_cond, omega, base_tol, tol));
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status batch_gmres_finish(kfbi_problem* p0, const ArnDesc* d, const BatchInst* inst, int n, const int* jdev,
                               const int* flags, cudaStream_t st) {
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_batch_finish<<<n, kBatchThreads, 0, st>>>(d, inst, jdev, flags));
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status batch_arnoldi_copy_in(kfbi_problem* p0, const ArnDesc* d, const int* jdev, const int* done,
                                  int ninst, int maxnb, cudaStream_t st) {
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_copy_in_batched<<<dim3(div_up(maxnb, 256), ninst), 256, 0, st>>>(d, jdev, done));
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status batch_arnoldi_step(kfbi_problem* p0, const ArnDesc* d, int* jdev, const int* done,
                               double* res_out, int ninst, int maxnb, int m, cudaStream_t st) {
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_copy_out_batched<<<dim3(div_up(maxnb, 256), ninst), 256, 0, st>>>(d, jdev, done));
  size_t smem = sizeof(double) * ((size_t)(m + 2) * (kArnThreads / 32) + 2 * (size_t)(m + 2));
  KFBI_LAUNCH(p0, KFBI_KC_GMRES, k_arnoldi_batched<<<ninst, kArnThreads, smem, st>>>(d, jdev, done, res_out));
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

// Initialise GMRES of instance p with zero start: V_0 = b/|b|, g = (|b|, 0, ...).
kfbi_status gmres_init_zero(kfbi_problem* p, const double* b, double bnorm) {
  Gmres& G = p->gm;
  cudaStream_t st = p->stream;
  const int eb = std::min(div_up(G.nb, 256), 152 * 4);
  KFBI_CUDA(p, cudaMemcpyAsync(G.scal, &bnorm, sizeof(double), cudaMemcpyHostToDevice, st));
  KFBI_CUDA(p, cudaMemcpyAsync(G.V, b, sizeof(double) * G.nb, cudaMemcpyDeviceToDevice, st));
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_scale<<<eb, 256, 0, st>>>(G.V, G.nb, G.scal, 1));
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_init_g<<<1, 128, 0, st>>>(G.g, G.m, G.scal));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status gmres_norm2(kfbi_problem* p, const double* v, double* out_dev) { return dot_self_pub(p, v, out_dev); }

// x = sum_{i < k} y_i V_i after solving H y = g (k x k)
kfbi_status gmres_finish(kfbi_problem* p, int k, double* x) {
  Gmres& G = p->gm;
  cudaStream_t st = p->stream;
  const int eb = std::min(div_up(G.nb, 256), 152 * 4);
  KFBI_CUDA(p, cudaMemsetAsync(x, 0, sizeof(double) * G.nb, st));
  if (k <= 0) return KFBI_OK;
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_solve_y<<<1, 1, 0, st>>>(G.H, G.m + 1, k, G.g, G.y));
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_update_x<<<eb, 256, 0, st>>>(G.V, G.nb, k, G.y, x));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status gmres_create(kfbi_problem* p, int m) {
  Gmres& G = p->gm;
  G.nb = p->nx;   // the BIE's unknowns (2 N_b for the general interface kind)
  G.m = m;
  G.nchunk = std::max(1, std::min(1024, div_up(G.nb, 2048)));
  KFBI_CUDA(p, dalloc(&G.V, (size_t)(m + 1) * G.nb));
  KFBI_CUDA(p, dalloc(&G.H, (size_t)(m + 1) * m));
  KFBI_CUDA(p, dalloc(&G.cs, m));
  KFBI_CUDA(p, dalloc(&G.sn, m));
  KFBI_CUDA(p, dalloc(&G.g, m + 1));
  KFBI_CUDA(p, dalloc(&G.y, m));
  KFBI_CUDA(p, dalloc(&G.part, (size_t)(m + 1) * G.nchunk));
  KFBI_CUDA(p, dalloc(&G.scal, 8));
  KFBI_CUDA(p, cudaMallocHost(reinterpret_cast<void**>(&G.host_res), 4 * sizeof(double)));
  KFBI_CUDA(p, dalloc(&G.jdev, 4));
  KFBI_CUDA(p, cudaMemset(G.jdev, 0, 4 * sizeof(int)));
  KFBI_CUDA(p, dalloc(&G.h1, m + 1));
  KFBI_CUDA(p, dalloc(&G.h2, m + 1));
  KFBI_CUDA(p, dalloc(&G.npart, 152 * 4));
  return KFBI_OK;
}

void gmres_destroy(kfbi_problem* p) {
  Gmres& G = p->gm;
  cudaFree(G.V);
  cudaFree(G.H);
  cudaFree(G.cs);
  cudaFree(G.sn);
  cudaFree(G.g);
  cudaFree(G.y);
  cudaFree(G.part);
  cudaFree(G.scal);
  if (G.host_res) cudaFreeHost(G.host_res);
  if (G.loop_exec) cudaGraphExecDestroy(G.loop_exec);
  if (G.loop_graph) cudaGraphDestroy(G.loop_graph);
  cudaFree(G.jdev);
  cudaFree(G.h1);
  cudaFree(G.h2);
  cudaFree(G.npart);
  G = Gmres();
}

// ||v||^2 into out[0] (device)
static kfbi_status dot_self(kfbi_problem* p, const double* v, double* out) { return dot_self_pub(p, v, out); }
kfbi_status dot_self_pub(kfbi_problem* p, const double* v, double* out) {
  Gmres& G = p->gm;
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_dots<<<dim3(G.nchunk, 1), kDotThreads, 0, p->stream>>>(v, G.nb, 1, v, G.nchunk, G.part));
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_reduce<<<1, kDotThreads, 0, p->stream>>>(G.part, G.nchunk, out, 0));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

static kfbi_status read_scalar(kfbi_problem* p, const double* dev, double* host) {
  KFBI_CUDA(p, cudaMemcpyAsync(p->gm.host_res, dev, sizeof(double), cudaMemcpyDeviceToHost, p->stream));
  KFBI_CUDA(p, cudaStreamSynchronize(p->stream));
  *host = p->gm.host_res[0];
  return KFBI_OK;
}

// The kernels of one GMRES iteration of problem p on its stream, V_j in the
// operator's input buffer: y = A x (the operator's kernels); CGS2 over all SMs,
// starting from y; norm, normalisation (V_{j+1} also into x) and Givens update;
// j <- j + 1.  With use_cond the finish kernel also sets the condition of the
// enclosing device-driven loop.  (Copies of V_j and y, the clearing of the
// right-hand side and of the boundary layer and a norm kernel of its own were
// five launches more: 64^2 Dirichlet solve 706 -> 677 us, 1024^2 mixed 3515 -> 3462.)
static kfbi_status iteration_body(kfbi_problem* p, cudaGraphConditionalHandle cond, int use_cond) {
  Gmres& G = p->gm;
  const int nb = G.nb;
  const int eb = std::min(div_up(nb, kCgsThreads), 152 * 4);
  KFBI_TRY(relax_box_tol(p));
  KFBI_TRY(apply_operator_impl(p, p->xbuf, p->ybuf));
  cudaStream_t cs = p->stream;
  const dim3 dg(G.nchunk, G.m + 1);
  for (int pass = 0; pass < 2; ++pass) {
    const double* y = pass ? nullptr : p->ybuf;
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_cgs_dots<<<dg, kCgsThreads, 0, cs>>>(G.V, nb, G.jdev, G.nchunk, y, G.part));
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_cgs_update<<<eb, kCgsThreads, 0, cs>>>(
        G.V, nb, G.jdev, G.part, G.nchunk, y, pass ? G.h2 : G.h1, pass ? G.npart : nullptr));
  }
  KFBI_LAUNCH(p, KFBI_KC_GMRES, k_cgs_finish<<<eb, kCgsThreads, 0, cs>>>(
      G.V, nb, p->xbuf, G.H, G.m + 1, G.cs, G.sn, G.g, G.scal + 2, G.h1, G.h2, G.npart, eb, G.jdev, cond, use_cond,
      G.scal + 5));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

// Capture iteration_body on the private stream, into `into` when given
// (cudaStreamBeginCaptureToGraph), else into a new graph returned in *out.
static kfbi_status capture_body(kfbi_problem* p, cudaGraph_t into, cudaGraph_t* out,
                                cudaGraphConditionalHandle cond, int use_cond) {
  Gmres& G = p->gm;
  cudaStream_t st = p->stream;
  if (!p->cap_stream) KFBI_CUDA(p, cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
  KFBI_CUDA(p, cudaStreamSynchronize(st));
  long long before[KFBI_KC_COUNT];
  for (int k = 0; k < KFBI_KC_COUNT; ++k) before[k] = p->prof.launches[k];
  const bool prof = p->prof.on;
  p->prof.on = false;
  set_stream(p, p->cap_stream);
  kfbi_status s = KFBI_OK;
  cudaError_t e = into ? cudaStreamBeginCaptureToGraph(p->cap_stream, into, nullptr, nullptr, 0,
                                                       cudaStreamCaptureModeThreadLocal)
                       : cudaStreamBeginCapture(p->cap_stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) s = iteration_body(p, cond, use_cond);
  cudaGraph_t gr = nullptr;
  cudaError_t e2 = e == cudaSuccess ? cudaStreamEndCapture(p->cap_stream, &gr) : e;
  set_stream(p, st);
  p->prof.on = prof;
  for (int k = 0; k < KFBI_KC_COUNT; ++k) {
    G.it_counts[k] = p->prof.launches[k] - before[k];
    p->prof.launches[k] = before[k];
  }
  if (e != cudaSuccess || e2 != cudaSuccess || s != KFBI_OK) {
    if (gr && !into) cudaGraphDestroy(gr);
    cudaGetLastError();
    return s != KFBI_OK ? s : fail(p, KFBI_ERR_CUDA, "GMRES iteration capture failed");
  }
  *out = gr;
  return KFBI_OK;
}

// The whole Arnoldi cycle on the device: a conditional WHILE node whose body is
// one iteration; the finish kernel ends the loop when the residual estimate
// reaches the threshold or after the iteration limit jdev[2], so the host
// synchronises once per cycle instead of once per iteration.  Returns false
// (the caller then launches the iterations one by one) if the driver refuses
// conditional nodes.
static bool loop_graph(kfbi_problem* p) {
  Gmres& G = p->gm;
  if (G.loop_exec) return true;
  if (G.loop_failed) return false;
  G.loop_failed = true;
  cudaGraph_t g = nullptr;
  if (cudaGraphCreate(&g, 0) != cudaSuccess) return false;
  cudaGraphConditionalHandle h;
  cudaGraphNodeParams np = {};
  cudaGraphNode_t node;
  bool ok = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
  if (ok) {
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    ok = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np) == cudaSuccess;
  }
  cudaGraph_t body = ok ? np.conditional.phGraph_out[0] : nullptr;
  cudaGraph_t captured = nullptr;
  if (ok) ok = capture_body(p, body, &captured, h, 1) == KFBI_OK;
  if (ok) ok = cudaGraphInstantiate(&G.loop_exec, g, 0) == cudaSuccess;
  if (!ok) {
    cudaGraphDestroy(g);
    cudaGetLastError();
    G.loop_exec = nullptr;
    return false;
  }
  G.loop_graph = g;
  G.loop_failed = false;
  return true;
}

kfbi_status gmres_run(kfbi_problem* p, const double* b, const double* x0, double rtol, int restart,
                      int max_iter, double* x, int* iters, double* rel, int* x0_rejected) {
  Gmres& G = p->gm;
  const int nb = G.nb;
  const int m = std::max(1, std::min(restart, G.m));
  cudaStream_t st = p->stream;
  const int eb = std::min(div_up(nb, 256), 152 * 4);
  double* beta = G.scal + 0;
  double* bn2 = G.scal + 1;
  double* res = G.scal + 2;
  KFBI_TRY(dot_self(p, b, bn2));
  double bnorm2;
  KFBI_TRY(read_scalar(p, bn2, &bnorm2));
  const double bnorm = std::sqrt(bnorm2);
  *iters = 0;
  *rel = 0.0;
  if (x0_rejected) *x0_rejected = 0;
  if (!std::isfinite(bnorm)) return fail(p, KFBI_ERR_NONFINITE, "non-finite BIE right-hand side");
  if (bnorm == 0.0) {
    KFBI_CUDA(p, cudaMemsetAsync(x, 0, sizeof(double) * nb, st));
    return KFBI_OK;
  }
  if (x0) {
    if (x0 != x) KFBI_CUDA(p, cudaMemcpyAsync(x, x0, sizeof(double) * nb, cudaMemcpyDeviceToDevice, st));
  } else {
    KFBI_CUDA(p, cudaMemsetAsync(x, 0, sizeof(double) * nb, st));
  }
  bool nonzero_x = x0 != nullptr;
  int total = 0;
  for (;;) {
    double* V0 = G.V;
    if (nonzero_x) {
      // the residual of a start or a restart at the full box-solve accuracy
      KFBI_TRY(box_tol_reset(p));
      if (p->twin) KFBI_TRY(box_tol_reset(p->twin));
      KFBI_TRY(apply_operator_fast(p, x, V0));
      KFBI_LAUNCH(p, KFBI_KC_GMRES, k_sub<<<eb, 256, 0, st>>>(b, V0, nb));
    } else {
      KFBI_CUDA(p, cudaMemcpyAsync(V0, b, sizeof(double) * nb, cudaMemcpyDeviceToDevice, st));
    }
    KFBI_TRY(dot_self(p, V0, beta));
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_sqrt<<<1, 1, 0, st>>>(beta));
    double hbeta;
    KFBI_TRY(read_scalar(p, beta, &hbeta));
    if (!std::isfinite(hbeta) && !(total == 0 && x0)) return fail(p, KFBI_ERR_NONFINITE, "non-finite GMRES residual");
    if (total == 0 && nonzero_x && x0 && !(hbeta < bnorm)) {
      // the initial guess is no better than zero: start from zero instead
      if (x0_rejected) *x0_rejected = 1;
      KFBI_CUDA(p, cudaMemsetAsync(x, 0, sizeof(double) * nb, st));
      nonzero_x = false;
      continue;
    }
    if (hbeta <= rtol * bnorm) {
      *iters = total;
      *rel = hbeta / bnorm;
      return KFBI_OK;
    }
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_scale<<<eb, 256, 0, st>>>(V0, nb, beta, 1));
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_init_g<<<1, 128, 0, st>>>(G.g, G.m, beta));
    KFBI_CUDA(p, cudaMemcpyAsync(p->xbuf, V0, sizeof(double) * nb, cudaMemcpyDeviceToDevice, st));
    // the residual estimate starts at beta and the threshold is rtol ||b||
    // (both read on the device by the loop and by the relaxation)
    {
      const double thr0 = rtol * bnorm;
      KFBI_CUDA(p, cudaMemcpyAsync(res, beta, sizeof(double), cudaMemcpyDeviceToDevice, st));
      KFBI_CUDA(p, cudaMemcpyAsync(G.scal + 5, &thr0, sizeof(double), cudaMemcpyHostToDevice, st));
    }
    int jend = 0;
    double hres = hbeta;
    const bool graph_it = p->use_graphs && !p->prof.on;
    if (graph_it && loop_graph(p)) {
      // one launch runs the cycle: at most min(m, max_iter - total) iterations
      const int jmax = std::min(m, max_iter - total);
      const int head[4] = {0, 0, jmax, 0};
      const double thr = rtol * bnorm;
      KFBI_CUDA(p, cudaMemcpyAsync(G.jdev, head, sizeof(head), cudaMemcpyHostToDevice, st));
      KFBI_CUDA(p, cudaMemcpyAsync(G.scal + 5, &thr, sizeof(double), cudaMemcpyHostToDevice, st));
      KFBI_CUDA(p, cudaGraphLaunch(G.loop_exec, st));
      int jdone = 0;
      KFBI_CUDA(p, cudaMemcpyAsync(G.host_res, res, sizeof(double), cudaMemcpyDeviceToHost, st));
      KFBI_CUDA(p, cudaMemcpyAsync(&jdone, G.jdev + 3, sizeof(int), cudaMemcpyDeviceToHost, st));
      KFBI_CUDA(p, cudaStreamSynchronize(st));
      hres = G.host_res[0];
      if (jdone < 1 || jdone > jmax) return fail(p, KFBI_ERR_CUDA, "device-driven GMRES loop lost its step count");
      for (int k = 0; k < KFBI_KC_COUNT; ++k) p->prof.launches[k] += G.it_counts[k] * jdone;
      total += jdone;
      jend = jdone;
      if (!std::isfinite(hres)) return fail(p, KFBI_ERR_NONFINITE, "non-finite GMRES residual");
    } else {
      KFBI_CUDA(p, cudaMemsetAsync(G.jdev, 0, 4 * sizeof(int), st));
      for (int j = 0; j < m; ++j) {
        KFBI_TRY(iteration_body(p, 0, 0));
        ++total;
        KFBI_TRY(read_scalar(p, res, &hres));
        jend = j + 1;
        if (!std::isfinite(hres)) return fail(p, KFBI_ERR_NONFINITE, "non-finite GMRES residual");
        if (hres <= rtol * bnorm || total >= max_iter) break;
      }
    }
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_solve_y<<<1, 1, 0, st>>>(G.H, G.m + 1, jend, G.g, G.y));
    KFBI_LAUNCH(p, KFBI_KC_GMRES, k_update_x<<<eb, 256, 0, st>>>(G.V, nb, jend, G.y, x));
    KFBI_CUDA(p, cudaGetLastError());
    nonzero_x = true;
    *iters = total;
    *rel = hres / bnorm;
    if (hres <= rtol * bnorm) {
      KFBI_CUDA(p, cudaStreamSynchronize(st));
      return KFBI_OK;
    }
    if (total >= max_iter)
      return fail(p, KFBI_ERR_NOT_CONVERGED,
                  "GMRES reached max_iter = " + std::to_string(max_iter) +
                      " (relative residual " + std::to_string(hres / bnorm) + ")");
  }
}

}  // namespace kfbi

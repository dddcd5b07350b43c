// Learned initial density for GMRES (Algorithm 1, Step 4 from a learned
// start instead of zero): a small fully connected network evaluated at every
// DOF, trained on the GPU on densities that the method itself computes.
//
//   z1 = W1 x + b1, a1 = tanh z1;  z2 = W2 a1 + b2, a2 = tanh z2;
//   y = W3 a2 + b3 + WL x
//
// Precision: FP32 master weights; the products with W1, W2, W3 use those
// weights rounded to bfloat16 (kept in a BF16 copy refreshed after each
// update); the linear skip WL, activations and all sums are FP32, so the
// linear part of the map is resolved beyond bfloat16 precision.  Gradients are those at the rounded weights and update the
// FP32 masters with Adam (Kingma & Ba 2015, bias-corrected moments).
//
// The contractions (K = 16 or 256, N = 256; the weight gradients K = rows) run
// on the tensor cores: mma.sync bf16 with FP32 accumulation, FP32 operands
// split into bf16 parts so that the products keep FP32 precision (k_gemm).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "kfbi_internal.cuh"

struct kfbi_mlp {
  int n_in = 0, width = 0, nparam = 0;
  int oW1 = 0, ob1 = 0, oW2 = 0, ob2 = 0, oW3 = 0, ob3 = 0, oWL = 0;
  cudaStream_t stream = nullptr;
  std::string err;
  float* theta = nullptr;          // FP32 masters
  float* grad = nullptr;
  float* mom1 = nullptr;
  float* mom2 = nullptr;
  __nv_bfloat16* wbf = nullptr;    // rounded copy, master layout
  float* shift = nullptr;          // [n_in] input normalisation x~ = (x - shift) * scale
  float* scale = nullptr;
  double out_shift = 0.0, out_scale = 1.0;
  long long step = 0;
  int train_lo = 0, train_hi = 0;  // parameters that Adam updates: [train_lo, train_hi)
  // per-row scratch
  int cap = 0;
  float* X = nullptr;     // normalised input [cap][n_in]
  float* a1 = nullptr;    // [cap][width]
  float* a2 = nullptr;
  float* d1 = nullptr;    // back-propagated signals [cap][width]
  float* d2 = nullptr;
  float* y = nullptr;     // [cap]
  float* tb = nullptr;    // gathered targets [cap]
  float* loss = nullptr;  // [1]
};

namespace kfbi {
namespace {

kfbi_status mfail(kfbi_mlp* m, kfbi_status s, const std::string& msg) {
  if (m) m->err = msg;
  return s;
}

#define MLP_CUDA(m, call)                                                         \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) return mfail((m), KFBI_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// ---- tensor-core GEMM: mma.sync m16n8k16, bf16 operands, FP32 accumulation --
// An FP32 operand enters as a sum of bfloat16 parts, x = hi + mid + lo with
// each part the bf16 rounding of what the previous parts leave; every product
// of two bf16 values is exact in FP32, so three parts carry an FP32 value's
// 24 bits.  Weights already rounded to bf16 are one exact part.
//
// C (M x N) = A (M x K) B (K x N), 64 x 64 tiles, four warps of 32 x 32 (2 x 4
// mma tiles), K in steps of 32; blockIdx.z splits K into chunks.  An operand is
// read along its contiguous axis (KC: the K axis, else its row or column
// axis), the next step's values into registers while this step's products run,
// cut into parts once, as they are stored to shared memory in pairs along K,
// and read back by ldmatrix (rows of 20 words: no bank conflicts).  The tile's
// products take 5 us of the tensor cores at 8192 x 256 x 256; a first version
// that staged FP32 values one K step of 16 at a time and cut them per warp ran
// at the memory latency of each step: 74 us, this one 26.
constexpr int kGT = 64, kGK = 32, kGP = 20;   // tile, K step, pitch in words (pairs of bf16)

__device__ __forceinline__ float gval(float v) { return v; }
__device__ __forceinline__ float gval(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void gvec4(const float* p, float* x) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  x[0] = v.x;
  x[1] = v.y;
  x[2] = v.z;
  x[3] = v.w;
}
__device__ __forceinline__ void gvec4(const __nv_bfloat16* p, float* x) {
  const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
  x[0] = __uint_as_float(v.x << 16);
  x[1] = __uint_as_float(v.x & 0xffff0000u);
  x[2] = __uint_as_float(v.y << 16);
  x[3] = __uint_as_float(v.y & 0xffff0000u);
}

// 16 values of this thread's share of a 64 x 32 operand tile (rows r0.., terms
// k0..; zero beyond R and ke).  KC: row r at p + r ld, four consecutive terms
// of four rows; else term k at p + k ld, four consecutive rows of two terms,
// twice.  vec: the groups of four are aligned and end with the operand.
template <bool KC, typename T>
__device__ __forceinline__ void g_load(const T* __restrict__ p, long long ld, int R, int ke, int r0, int k0, bool vec,
                                       float (&x)[16]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int r = KC ? r0 + (tid >> 3) + 16 * it : r0 + 4 * ((tid >> 4) + 8 * (it >> 1));
    const int k = KC ? k0 + 4 * (tid & 7) : k0 + 2 * (tid & 15) + (it & 1);
    float* v = x + 4 * it;
    const T* q = KC ? p + r * ld + k : p + k * ld + r;
    if (vec) {
      if (r < R && k < ke) {
        gvec4(q, v);
      } else {
        v[0] = v[1] = v[2] = v[3] = 0.f;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool ok = KC ? r < R && k + e < ke : r + e < R && k < ke;
        v[e] = ok ? gval(q[e]) : 0.f;
      }
    }
  }
}

// the pair (a, b), b in the upper half, as PARTS bf16 words
template <int PARTS>
__device__ __forceinline__ void g_split(float a, float b, uint32_t (&w)[PARTS]) {
#pragma unroll
  for (int q = 0; q < PARTS; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    w[q] = *reinterpret_cast<const uint32_t*>(&h);
    a -= __uint_as_float(w[q] << 16);
    b -= __uint_as_float(w[q] & 0xffff0000u);
  }
}

template <bool KC, int PARTS>
__device__ __forceinline__ void g_store(uint32_t* s, const float (&x)[16]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int it = 0; it < (KC ? 4 : 2); ++it) {
    if (KC) {
      uint32_t w0[PARTS], w1[PARTS];
      g_split<PARTS>(x[4 * it], x[4 * it + 1], w0);
      g_split<PARTS>(x[4 * it + 2], x[4 * it + 3], w1);
      const int at = ((tid >> 3) + 16 * it) * kGP + 2 * (tid & 7);
#pragma unroll
      for (int q = 0; q < PARTS; ++q)
        *reinterpret_cast<uint2*>(s + q * kGT * kGP + at) = make_uint2(w0[q], w1[q]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t w[PARTS];
        g_split<PARTS>(x[8 * it + e], x[8 * it + 4 + e], w);
        const int at = (4 * ((tid >> 4) + 8 * it) + e) * kGP + (tid & 15);
#pragma unroll
        for (int q = 0; q < PARTS; ++q) s[q * kGT * kGP + at] = w[q];
      }
    }
  }
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const uint32_t* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// mode 0: C = act(acc + bias) [* (1 - gate^2)], and csum_j += sum_i C_ij;
// mode 1: C += acc (atomic).
template <bool AKC, bool BKC, typename TB>
__global__ void __launch_bounds__(128) k_gemm(int M, int N, int K, int kchunk, const float* __restrict__ A,
                                              long long lda, bool avec, const TB* __restrict__ B, long long ldb,
                                              bool bvec, float* __restrict__ C, long long ldc,
                                              const float* __restrict__ bias, int act, const float* __restrict__ gate,
                                              float* __restrict__ csum, int mode) {
  constexpr int BP = sizeof(TB) == 2 ? 1 : 3;
  __shared__ __align__(16) uint32_t As[3 * kGT * kGP];
  __shared__ __align__(16) uint32_t Bs[BP * kGT * kGP];
  const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT;
  const int kb = blockIdx.z * kchunk;
  const int ke = min(K, kb + kchunk);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tq = lane & 3;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  float acc[2][4][4];
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[mi][ni][e] = 0.f;
  float ra[16], rb[16];
  g_load<AKC>(A, lda, M, ke, m0, kb, avec, ra);
  g_load<BKC>(B, ldb, N, ke, n0, kb, bvec, rb);
  const uint32_t* pa = As + (wm + (lane & 15)) * kGP + 4 * (lane >> 4);
  const uint32_t* pb = Bs + (wn + (lane & 7) + 8 * (lane >> 4)) * kGP + 4 * ((lane >> 3) & 1);
  for (int k0 = kb; k0 < ke; k0 += kGK) {
    g_store<AKC, 3>(As, ra);
    g_store<BKC, BP>(Bs, rb);
    __syncthreads();
    if (k0 + kGK < ke) {
      g_load<AKC>(A, lda, M, ke, m0, k0 + kGK, avec, ra);
      g_load<BKC>(B, ldb, N, ke, n0, k0 + kGK, bvec, rb);
    }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      if (kk == 1 && k0 + 16 >= ke) break;
      uint32_t af[3][2][4];
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int mi = 0; mi < 2; ++mi) ldsm4(af[q][mi], pa + (q * kGT + mi * 16) * kGP + 8 * kk);
#pragma unroll
      for (int nj = 0; nj < 2; ++nj) {
        uint32_t bf[BP][4];
#pragma unroll
        for (int q = 0; q < BP; ++q) ldsm4(bf[q], pb + (q * kGT + nj * 16) * kGP + 8 * kk);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int mi = 0; mi < 2; ++mi) {
            float* c = acc[mi][2 * nj + h];
            // small terms first: lo, mid, then hi
            if (BP == 1) {
              mma16816(c, af[2][mi], bf[0] + 2 * h);
              mma16816(c, af[1][mi], bf[0] + 2 * h);
              mma16816(c, af[0][mi], bf[0] + 2 * h);
            } else {
              mma16816(c, af[2][mi], bf[0] + 2 * h);
              mma16816(c, af[0][mi], bf[BP - 1] + 2 * h);
              mma16816(c, af[1][mi], bf[BP / 2] + 2 * h);
              mma16816(c, af[1][mi], bf[0] + 2 * h);
              mma16816(c, af[0][mi], bf[BP / 2] + 2 * h);
              mma16816(c, af[0][mi], bf[0] + 2 * h);
            }
          }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int ni = 0; ni < 4; ++ni) {
    const int j = n0 + wn + ni * 8 + 2 * tq;
    float cs[2] = {0.f, 0.f};
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int i = m0 + wm + mi * 16 + g + (e >= 2 ? 8 : 0);
        const int jj = j + (e & 1);
        if (i >= M || jj >= N) continue;
        float* o = C + (long long)i * ldc + jj;
        if (mode == 1) {
          atomicAdd(o, acc[mi][ni][e]);
        } else {
          float v = acc[mi][ni][e] + (bias ? bias[jj] : 0.f);
          if (act) v = tanhf(v);
          if (gate) {
            const float gt = gate[(long long)i * ldc + jj];
            v *= 1.f - gt * gt;
          }
          *o = v;
          cs[e & 1] += v;
        }
      }
    if (csum) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) cs[e] += __shfl_xor_sync(0xffffffffu, cs[e], o);
        if (g == 0 && j + e < N) atomicAdd(csum + j + e, cs[e]);
      }
    }
  }
}

// X[i, :] = (raw[r_i, :] - shift) * scale with r_i = rows[i] (i when rows is
// null); the targets of the selected rows are gathered alongside.
__global__ void k_normalise(int n, int n_in, const float* __restrict__ raw, const int32_t* __restrict__ rows,
                            const float* __restrict__ shift, const float* __restrict__ scale,
                            float* __restrict__ X, const float* __restrict__ t_in, float* __restrict__ t_out) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)n * n_in) return;
  const int k = (int)(t % n_in);
  const long long i = t / n_in;
  const long long r = rows ? (long long)rows[i] : i;
  X[t] = (raw[r * n_in + k] - shift[k]) * scale[k];
  if (t_in && k == 0) t_out[i] = t_in[r];
}

// y_i = W3 a2_i + b3 + WL x_i (a warp per row)
__device__ __forceinline__ float row_output(int W, const float* __restrict__ a, const __nv_bfloat16* __restrict__ w3,
                                            float b3, int n_in, const float* __restrict__ x,
                                            const float* __restrict__ wl) {
  const int lane = threadIdx.x & 31;
  float s = 0.f;
  for (int k = lane; k < W; k += 32) s = fmaf(a[k], __bfloat162float(w3[k]), s);
  if (lane < n_in) s = fmaf(x[lane], wl[lane], s);
  return warp_sum(s) + b3;
}

__global__ void k_output(int n, int W, const float* __restrict__ a2, const __nv_bfloat16* __restrict__ w3,
                         const float* __restrict__ b3, int n_in, const float* __restrict__ X,
                         const float* __restrict__ wl, float* __restrict__ y) {
  const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (row >= n) return;
  const float v = row_output(W, a2 + (long long)row * W, w3, b3[0], n_in, X + (long long)row * n_in, wl);
  if ((threadIdx.x & 31) == 0) y[row] = v;
}

// The head of a training step over kHeadRows rows per CTA: the outputs, the
// loss 1/(2n) sum e^2, dy = e/n, the back-propagated d2 = dy W3 (1 - a2^2), and
// the gradients of the output layer and of b2 (dW3 = dy^T a2, db3 = sum dy, dWL =
// dy^T x~, db2 = sum d2), one pass over a2 with a column per thread.  Six
// launches, four of them column sums of 32 CTAs that waited on one load per
// row, took 119 us for 8192 rows; this kernel 16.
constexpr int kHeadRows = 32, kHeadThreads = 256;
__global__ void __launch_bounds__(kHeadThreads) k_head(int n, int W, const float* __restrict__ a2,
                                                       const __nv_bfloat16* __restrict__ w3,
                                                       const float* __restrict__ b3, int n_in,
                                                       const float* __restrict__ X, const float* __restrict__ wl,
                                                       const float* __restrict__ t, float* __restrict__ y,
                                                       float* __restrict__ d2, float* __restrict__ loss,
                                                       float* __restrict__ gW3, float* __restrict__ gb3,
                                                       float* __restrict__ gWL, float* __restrict__ gb2) {
  __shared__ float dy[kHeadRows];
  __shared__ float es[kHeadThreads / 32];
  const int r0 = blockIdx.x * kHeadRows, nr = min(kHeadRows, n - r0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float e2 = 0.f;
  for (int r = warp; r < kHeadRows; r += kHeadThreads / 32) {
    float e = 0.f;
    if (r < nr) {
      const long long row = r0 + r;
      const float v = row_output(W, a2 + row * W, w3, b3[0], n_in, X + row * n_in, wl);
      e = v - t[row];
      if (lane == 0) y[row] = v;
    }
    if (lane == 0) dy[r] = e / (float)n;
    e2 += e * e;
  }
  if (lane == 0) es[warp] = e2;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int q = 0; q < kHeadThreads / 32; ++q) s += es[q];
    atomicAdd(loss, 0.5f * s / (float)n);
  }
  for (int k = threadIdx.x; k < W; k += kHeadThreads) {
    const float w = __bfloat162float(w3[k]);
    const float* a = a2 + (long long)r0 * W + k;
    float* d = d2 + (long long)r0 * W + k;
    float s3 = 0.f, s2 = 0.f;
#pragma unroll 8
    for (int r = 0; r < nr; ++r) {
      const float v = a[(long long)r * W];
      const float b = dy[r] * w * (1.f - v * v);
      d[(long long)r * W] = b;
      s3 = fmaf(dy[r], v, s3);
      s2 += b;
    }
    atomicAdd(gW3 + k, s3);
    atomicAdd(gb2 + k, s2);
  }
  if (threadIdx.x <= n_in) {
    const int k = threadIdx.x;
    float s = 0.f;
    for (int r = 0; r < nr; ++r) s = fmaf(dy[r], k < n_in ? X[(long long)(r0 + r) * n_in + k] : 1.f, s);
    atomicAdd(k < n_in ? gWL + k : gb3, s);
  }
}

__global__ void k_round(int np, const float* __restrict__ theta, __nv_bfloat16* __restrict__ wbf) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < np) wbf[t] = __float2bfloat16_rn(theta[t]);
}

__global__ void k_adam(int lo, int hi, float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float bc1, float bc2,
                       __nv_bfloat16* __restrict__ wbf) {
  const int t = lo + blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= hi) return;
  const float gt = g[t];
  const float mt = b1 * m[t] + (1.f - b1) * gt;
  const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
  m[t] = mt;
  v[t] = vt;
  const float th = theta[t] - lr * (mt / bc1) / (sqrtf(vt / bc2) + eps);
  theta[t] = th;
  wbf[t] = __float2bfloat16_rn(th);
}

// Per-DOF raw features: [g1, g2, n (3), x (3), level-set parameters p0..p5,
// log10(sigma_in/sigma_out) (0 for a boundary value problem), 0].  The data
// are not rescaled per problem: the network's input normalisation (from its
// training set) brings each feature to unit size, and a problem family whose
// data share fields (the same sources with different geometries and
// coefficients) keeps its density a function of the DOF's features alone.
__global__ void k_features(int nb, int d, const double* __restrict__ x0, const double* __restrict__ x1,
                           const double* __restrict__ x2, const double* __restrict__ n0,
                           const double* __restrict__ n1, const double* __restrict__ n2,
                           const double* __restrict__ g1, const double* __restrict__ g2, LevelSet ls,
                           float lcontrast, float* __restrict__ F, const double* __restrict__ dens,
                           float* __restrict__ target) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nb) return;
  if (target) target[j] = (float)dens[j];
  float* f = F + (long long)j * KFBI_WS_FEATURES;
  f[0] = g1 ? (float)g1[j] : 0.f;
  f[1] = g2 ? (float)g2[j] : 0.f;
  f[2] = (float)n0[j];
  f[3] = (float)n1[j];
  f[4] = d == 3 ? (float)n2[j] : 0.f;
  f[5] = (float)x0[j];
  f[6] = (float)x1[j];
  f[7] = d == 3 ? (float)x2[j] : 0.f;
  for (int k = 0; k < 6; ++k) f[8 + k] = k < ls.np ? (float)ls.p[k] : 0.f;
  f[14] = lcontrast;
  f[15] = 0.f;
}

__global__ void k_to_density(int n, const float* __restrict__ y, double shift, double scale,
                             double* __restrict__ x) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) x[j] = (double)y[j] * scale + shift;
}

kfbi_status ensure(kfbi_mlp* m, int n) {
  if (n <= m->cap) return KFBI_OK;
  MLP_CUDA(m, cudaStreamSynchronize(m->stream));
  float** bufs[] = {&m->X, &m->a1, &m->a2, &m->d1, &m->d2, &m->y, &m->tb};
  for (float** b : bufs) {
    cudaFree(*b);
    *b = nullptr;
  }
  const int cap = std::max(n, 1024);
  const size_t W = m->width;
  MLP_CUDA(m, dalloc(&m->X, (size_t)cap * m->n_in));
  MLP_CUDA(m, dalloc(&m->a1, (size_t)cap * W));
  MLP_CUDA(m, dalloc(&m->a2, (size_t)cap * W));
  MLP_CUDA(m, dalloc(&m->d1, (size_t)cap * W));
  MLP_CUDA(m, dalloc(&m->d2, (size_t)cap * W));
  MLP_CUDA(m, dalloc(&m->y, (size_t)cap));
  MLP_CUDA(m, dalloc(&m->tb, (size_t)cap));
  m->cap = cap;
  return KFBI_OK;
}

// AKC / BKC: the operand is contiguous along K (A: M x K row-major, B: N x K),
// else along its other axis (A: K x M, B: K x N)
template <bool AKC, bool BKC, typename TB>
void gemm(cudaStream_t st, int M, int N, int K, const float* A, long long lda, const TB* B, long long ldb, float* C,
          long long ldc, const float* bias, int act, const float* gate, float* csum, int mode) {
  int splits = 1, chunk = K;
  if (mode == 1) {
    // weight gradients: long K (the rows), few output tiles.  Chunks of at
    // most 256 terms bound the rounding of one accumulator; few tiles (dW1) take
    // down to 128 for two CTAs per SM
    const int tiles = div_up(M, kGT) * div_up(N, kGT);
    splits = std::max(div_up(K, 256), std::min(div_up(K, 128), div_up(152 * 2, tiles)));
    chunk = div_up(div_up(K, splits), kGK) * kGK;
    splits = div_up(K, chunk);
  }
  auto vec = [](const void* p, size_t el, long long ld, int along) {
    return (reinterpret_cast<uintptr_t>(p) % (4 * el)) == 0 && ld % 4 == 0 && along % 4 == 0;
  };
  const bool av = vec(A, sizeof(float), lda, AKC ? K : M), bv = vec(B, sizeof(TB), ldb, BKC ? K : N);
  dim3 grid(div_up(N, kGT), div_up(M, kGT), splits);
  k_gemm<AKC, BKC, TB><<<grid, 128, 0, st>>>(M, N, K, chunk, A, lda, av, B, ldb, bv, C, ldc, bias, act, gate, csum,
                                              mode);
}

// the hidden layers of the rows already normalised into m->X
void hidden_rows(kfbi_mlp* m, int n) {
  const int W = m->width, ni = m->n_in;
  const __nv_bfloat16* wb = m->wbf;
  gemm<true, true>(m->stream, n, W, ni, m->X, ni, wb + m->oW1, ni, m->a1, W, m->theta + m->ob1, 1, nullptr, nullptr, 0);
  gemm<true, true>(m->stream, n, W, W, m->a1, W, wb + m->oW2, W, m->a2, W, m->theta + m->ob2, 1, nullptr, nullptr, 0);
}

// forward on rows already normalised into m->X
kfbi_status forward_rows(kfbi_mlp* m, int n) {
  hidden_rows(m, n);
  k_output<<<div_up(n, 8), 256, 0, m->stream>>>(n, m->width, m->a2, m->wbf + m->oW3, m->theta + m->ob3, m->n_in, m->X,
                                                m->theta + m->oWL, m->y);
  MLP_CUDA(m, cudaGetLastError());
  return KFBI_OK;
}

}  // namespace
}  // namespace kfbi

using namespace kfbi;

extern "C" {

const char* kfbi_mlp_last_error(const kfbi_mlp* m) { return m ? m->err.c_str() : ""; }

kfbi_status kfbi_mlp_destroy(kfbi_mlp* m) {
  if (!m) return KFBI_OK;
  if (m->stream) cudaStreamSynchronize(m->stream);
  void* bufs[] = {m->theta, m->grad, m->mom1, m->mom2, m->wbf, m->shift, m->scale, m->X,
                  m->a1,    m->a2,   m->d1,   m->d2,   m->y,   m->tb,   m->loss};
  for (void* b : bufs) cudaFree(b);
  delete m;
  return KFBI_OK;
}

kfbi_status kfbi_mlp_create(int n_in, int width, void* cuda_stream, kfbi_mlp** out) {
  if (!out || n_in < 1 || n_in > KFBI_WS_FEATURES || width < 1 || width > 1024) return KFBI_ERR_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return KFBI_ERR_CUDA;
  kfbi_mlp* m = new kfbi_mlp();
  m->n_in = n_in;
  m->width = width;
  m->stream = static_cast<cudaStream_t>(cuda_stream);
  m->oW1 = 0;
  m->ob1 = width * n_in;
  m->oW2 = m->ob1 + width;
  m->ob2 = m->oW2 + width * width;
  m->oW3 = m->ob2 + width;
  m->ob3 = m->oW3 + width;
  m->oWL = m->ob3 + 1;
  m->nparam = m->oWL + n_in;
  m->train_lo = 0;
  m->train_hi = m->nparam;
  const size_t np = m->nparam;
  bool ok = dalloc(&m->theta, np) == cudaSuccess && dalloc(&m->grad, np) == cudaSuccess &&
            dalloc(&m->mom1, np) == cudaSuccess && dalloc(&m->mom2, np) == cudaSuccess &&
            dalloc(&m->wbf, np) == cudaSuccess && dalloc(&m->shift, n_in) == cudaSuccess &&
            dalloc(&m->scale, n_in) == cudaSuccess && dalloc(&m->loss, 1) == cudaSuccess;
  if (ok) {
    std::vector<float> one(n_in, 1.f);
    ok = cudaMemset(m->theta, 0, np * 4) == cudaSuccess && cudaMemset(m->mom1, 0, np * 4) == cudaSuccess &&
         cudaMemset(m->mom2, 0, np * 4) == cudaSuccess && cudaMemset(m->grad, 0, np * 4) == cudaSuccess &&
         cudaMemset(m->wbf, 0, np * 2) == cudaSuccess && cudaMemset(m->shift, 0, n_in * 4) == cudaSuccess &&
         cudaMemcpy(m->scale, one.data(), n_in * 4, cudaMemcpyHostToDevice) == cudaSuccess;
  }
  if (!ok) {
    kfbi_mlp_destroy(m);
    return KFBI_ERR_CUDA;
  }
  *out = m;
  return KFBI_OK;
}

kfbi_status kfbi_mlp_num_params(const kfbi_mlp* m, int* count) {
  if (!m || !count) return KFBI_ERR_ARG;
  *count = m->nparam;
  return KFBI_OK;
}

kfbi_status kfbi_mlp_set_params(kfbi_mlp* m, const float* params) {
  if (!m || !params) return KFBI_ERR_ARG;
  MLP_CUDA(m, cudaMemcpyAsync(m->theta, params, sizeof(float) * m->nparam, cudaMemcpyDeviceToDevice, m->stream));
  MLP_CUDA(m, cudaMemsetAsync(m->mom1, 0, sizeof(float) * m->nparam, m->stream));
  MLP_CUDA(m, cudaMemsetAsync(m->mom2, 0, sizeof(float) * m->nparam, m->stream));
  m->step = 0;
  k_round<<<div_up(m->nparam, 256), 256, 0, m->stream>>>(m->nparam, m->theta, m->wbf);
  MLP_CUDA(m, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status kfbi_mlp_set_trainable(kfbi_mlp* m, int groups) {
  if (!m || groups < 0 || groups > 3) return KFBI_ERR_ARG;
  // the nonlinear branch [W1, b1, W2, b2, W3] precedes the linear part [b3, WL]
  m->train_lo = (groups & 1) ? 0 : m->ob3;
  m->train_hi = (groups & 2) ? m->nparam : m->ob3;
  if (groups == 0) m->train_lo = m->train_hi = 0;
  MLP_CUDA(m, cudaMemsetAsync(m->mom1, 0, sizeof(float) * m->nparam, m->stream));
  MLP_CUDA(m, cudaMemsetAsync(m->mom2, 0, sizeof(float) * m->nparam, m->stream));
  m->step = 0;
  return KFBI_OK;
}

kfbi_status kfbi_mlp_get_params(const kfbi_mlp* mc, float* params, float* grads) {
  kfbi_mlp* m = const_cast<kfbi_mlp*>(mc);
  if (!m) return KFBI_ERR_ARG;
  if (params)
    MLP_CUDA(m, cudaMemcpyAsync(params, m->theta, sizeof(float) * m->nparam, cudaMemcpyDeviceToDevice, m->stream));
  if (grads)
    MLP_CUDA(m, cudaMemcpyAsync(grads, m->grad, sizeof(float) * m->nparam, cudaMemcpyDeviceToDevice, m->stream));
  return KFBI_OK;
}

kfbi_status kfbi_mlp_set_affine(kfbi_mlp* m, const float* in_shift, const float* in_scale, double out_shift,
                                double out_scale) {
  if (!m || !in_shift || !in_scale || !std::isfinite(out_shift) || !std::isfinite(out_scale)) return KFBI_ERR_ARG;
  MLP_CUDA(m, cudaMemcpy(m->shift, in_shift, sizeof(float) * m->n_in, cudaMemcpyHostToDevice));
  MLP_CUDA(m, cudaMemcpy(m->scale, in_scale, sizeof(float) * m->n_in, cudaMemcpyHostToDevice));
  m->out_shift = out_shift;
  m->out_scale = out_scale;
  return KFBI_OK;
}

kfbi_status kfbi_mlp_forward(kfbi_mlp* m, const float* X, int n, float* y) {
  if (!m || n < 0 || (n > 0 && (!X || !y))) return KFBI_ERR_ARG;
  if (n == 0) return KFBI_OK;
  KFBI_TRY(ensure(m, n));
  const long long tot = (long long)n * m->n_in;
  k_normalise<<<div_up(tot, 256), 256, 0, m->stream>>>(n, m->n_in, X, nullptr, m->shift, m->scale, m->X,
                                                        nullptr, nullptr);
  KFBI_TRY(forward_rows(m, n));
  MLP_CUDA(m, cudaMemcpyAsync(y, m->y, sizeof(float) * n, cudaMemcpyDeviceToDevice, m->stream));
  return KFBI_OK;
}

kfbi_status kfbi_mlp_loss_grad(kfbi_mlp* m, const float* X, const float* t, const int32_t* rows, int n,
                               float* loss) {
  if (!m || !X || !t || n < 1) return KFBI_ERR_ARG;
  KFBI_TRY(ensure(m, n));
  cudaStream_t st = m->stream;
  const int W = m->width, ni = m->n_in;
  const long long tot = (long long)n * ni;
  MLP_CUDA(m, cudaMemsetAsync(m->loss, 0, sizeof(float), st));
  MLP_CUDA(m, cudaMemsetAsync(m->grad, 0, sizeof(float) * m->nparam, st));
  k_normalise<<<div_up(tot, 256), 256, 0, st>>>(n, ni, X, rows, m->shift, m->scale, m->X, t, m->tb);
  hidden_rows(m, n);
  const __nv_bfloat16* wb = m->wbf;
  float* g = m->grad;
  k_head<<<div_up(n, kHeadRows), kHeadThreads, 0, st>>>(n, W, m->a2, wb + m->oW3, m->theta + m->ob3, ni, m->X,
                                                        m->theta + m->oWL, m->tb, m->y, m->d2, m->loss, g + m->oW3,
                                                        g + m->ob3, g + m->oWL, g + m->ob2);
  // dW2 = d2^T a1; d1 = (d2 W2) (1 - a1^2), db1 = sum d1; dW1 = d1^T x~
  gemm<false, false>(st, W, W, n, m->d2, W, m->a1, W, g + m->oW2, W, nullptr, 0, nullptr, nullptr, 1);
  gemm<true, false>(st, n, W, W, m->d2, W, wb + m->oW2, W, m->d1, W, nullptr, 0, m->a1, g + m->ob1, 0);
  gemm<false, false>(st, W, ni, n, m->d1, W, m->X, ni, g + m->oW1, ni, nullptr, 0, nullptr, nullptr, 1);
  MLP_CUDA(m, cudaGetLastError());
  if (loss) MLP_CUDA(m, cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  return KFBI_OK;
}

kfbi_status kfbi_mlp_adam(kfbi_mlp* m, float lr, float beta1, float beta2, float eps) {
  if (!m || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) return KFBI_ERR_ARG;
  m->step += 1;
  const float bc1 = (float)(1.0 - std::pow((double)beta1, (double)m->step));
  const float bc2 = (float)(1.0 - std::pow((double)beta2, (double)m->step));
  const int cnt = m->train_hi - m->train_lo;
  if (cnt <= 0) return KFBI_OK;
  k_adam<<<div_up(cnt, 256), 256, 0, m->stream>>>(m->train_lo, m->train_hi, m->theta, m->grad, m->mom1, m->mom2,
                                                   lr, beta1, beta2, eps, bc1, bc2, m->wbf);
  MLP_CUDA(m, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status kfbi_warm_start_features(kfbi_problem* p, const kfbi_data* data, const double* density,
                                     float* features, float* target) {
  if (!p || !data || !features || !data->g1 || (!density != !target)) return KFBI_ERR_ARG;
  const Grid g = p->g;
  const bool iface = p->cfg.kind == KFBI_INTERFACE_MU || p->cfg.kind == KFBI_INTERFACE_GENERAL;
  const float lcontrast = iface ? (float)std::log10(p->cfg.sigma_in / p->cfg.sigma_out) : 0.f;
  KFBI_LAUNCH(p, KFBI_KC_OTHER, k_features<<<div_up(p->nb, 128), 128, 0, p->stream>>>(
      p->nb, g.d, p->x[0], p->x[1], g.d == 3 ? p->x[2] : p->x[0], p->nrm[0], p->nrm[1],
      g.d == 3 ? p->nrm[2] : p->nrm[0], data->g1, data->g2, p->ls, lcontrast, features, density, target));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status kfbi_warm_start(kfbi_problem* p, kfbi_mlp* m, const kfbi_data* data, double* x0) {
  if (!p || !m || !data || !x0 || !data->g1) return KFBI_ERR_ARG;
  if (p->nx != p->nb) return fail(p, KFBI_ERR_UNSUPPORTED, "the learned start predicts one density per DOF");
  if (m->n_in != KFBI_WS_FEATURES) return fail(p, KFBI_ERR_ARG, "the network must take KFBI_WS_FEATURES inputs");
  if (m->stream != p->stream) return fail(p, KFBI_ERR_ARG, "network and problem must share a stream");
  if (m->width < KFBI_WS_FEATURES) return fail(p, KFBI_ERR_ARG, "the network width must be >= KFBI_WS_FEATURES");
  const int nb = p->nb;
  {
    kfbi_status s = ensure(m, nb);
    if (s != KFBI_OK) return fail(p, s, m->err);
  }
  // features straight into the network's input scratch, then normalise in place
  KFBI_TRY(kfbi_warm_start_features(p, data, nullptr, m->d1, nullptr));
  const long long tot = (long long)nb * m->n_in;
  KFBI_LAUNCH(p, KFBI_KC_OTHER, k_normalise<<<div_up(tot, 256), 256, 0, p->stream>>>(
      nb, m->n_in, m->d1, nullptr, m->shift, m->scale, m->X, nullptr, nullptr));
  {
    kfbi_status s = forward_rows(m, nb);
    if (s != KFBI_OK) return fail(p, s, m->err);
  }
  KFBI_LAUNCH(p, KFBI_KC_OTHER, k_to_density<<<div_up(nb, 256), 256, 0, p->stream>>>(nb, m->y, m->out_shift,
                                                                                         m->out_scale, x0));
  KFBI_CUDA(p, cudaGetLastError());
  return KFBI_OK;
}

kfbi_status kfbi_warm_start_batch(kfbi_batch* b, kfbi_mlp* m, const kfbi_data* data, double* const* x0s) {
  if (!b || !m || !data || !x0s) return KFBI_ERR_ARG;
  const int n = batch_size(b);
  kfbi_problem* p0 = batch_problem(b, 0);
  if (m->n_in != KFBI_WS_FEATURES) return fail(p0, KFBI_ERR_ARG, "the network must take KFBI_WS_FEATURES inputs");
  if (m->stream != p0->stream) return fail(p0, KFBI_ERR_ARG, "network and batch must share a stream");
  if (m->width < KFBI_WS_FEATURES) return fail(p0, KFBI_ERR_ARG, "the network width must be >= KFBI_WS_FEATURES");
  std::vector<long long> off(n + 1, 0);
  for (int k = 0; k < n; ++k) {
    kfbi_problem* p = batch_problem(b, k);
    if (!x0s[k] || !data[k].g1) return fail(p0, KFBI_ERR_ARG, "missing data or start for an instance");
    if (p->nx != p->nb) return fail(p0, KFBI_ERR_UNSUPPORTED, "the learned start predicts one density per DOF");
    off[k + 1] = off[k] + p->nb;
  }
  if (off[n] > INT32_MAX / KFBI_WS_FEATURES) return fail(p0, KFBI_ERR_UNSUPPORTED, "too many DOFs in the batch");
  const int rows = (int)off[n];
  {
    kfbi_status s = ensure(m, rows);
    if (s != KFBI_OK) return fail(p0, s, m->err);
  }
  // every instance's features into one matrix, one normalisation and one
  // forward pass over all rows, then each instance's densities
  for (int k = 0; k < n; ++k)
    KFBI_TRY(kfbi_warm_start_features(batch_problem(b, k), &data[k], nullptr, m->d1 + off[k] * m->n_in, nullptr));
  const long long tot = (long long)rows * m->n_in;
  KFBI_LAUNCH(p0, KFBI_KC_OTHER, k_normalise<<<div_up(tot, 256), 256, 0, p0->stream>>>(
      rows, m->n_in, m->d1, nullptr, m->shift, m->scale, m->X, nullptr, nullptr));
  {
    kfbi_status s = forward_rows(m, rows);
    if (s != KFBI_OK) return fail(p0, s, m->err);
  }
  for (int k = 0; k < n; ++k) {
    const int nb = batch_problem(b, k)->nb;
    KFBI_LAUNCH(p0, KFBI_KC_OTHER, k_to_density<<<div_up(nb, 256), 256, 0, p0->stream>>>(
        nb, m->y + off[k], m->out_shift, m->out_scale, x0s[k]));
  }
  KFBI_CUDA(p0, cudaGetLastError());
  return KFBI_OK;
}

}  // extern "C"

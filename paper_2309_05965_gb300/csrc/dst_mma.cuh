// FP64 sine-transform passes as exact integer matrix products on the tensor
// cores.  Included by dst.cu (uses its PassArgs and fixed-point helpers).
//
// GB300 runs FP64 at 2 lanes per clock per SM, so an FP64 FFT pass is bound by
// that pipe whatever its layout (the radix-4 pass of dst.cu spends 72 % of
// its time there).  The tensor cores multiply FP16 integers exactly, so a
// DST-I of N - 1 points runs here as a matrix product in fixed point (the
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012):
//   * each line is scaled by a power of two to 60-bit integers (its largest
//     element decides), the matrix S_kj = sin(pi k j / N) is held to 62 bits;
//   * two exact foldings x_j +- x_{N-j} separate the modes k odd (K = N/2
//     terms), k = 2 mod 4 and k = 0 mod 4 (K = N/4 each): 3/8 of the dense
//     products;
//   * both factors are cut into 8 balanced base-256 digits (FP16 holds them
//     exactly); products of digits i + j = d <= 7 are summed over K <= 128
//     terms in one FP32 accumulator per d, exactly: 8 * 128 * 2^14 = 2^24;
//   * the eight sums are put together in 64-bit integers and rounded once to
//     FP64.  The dropped products i + j >= 8 are at most about 7 2^14 2^48 per
//     term, 2^-57 of the line's largest element (the unit 2^122), so 2^-48 over 512
//     terms; digits of no pattern leave about 2^-55.  Measured, the result is
//     closer to the exact transform than an FP64 FFT's (the launch rule in dst.cu).
#pragma once
#include <cooperative_groups.h>
#include <cuda_fp16.h>

namespace kfbi {
namespace {

constexpr int kMmaMinN = 64, kMmaMaxN2 = 1024, kMmaMaxN3 = 512;   // box sizes the kernel takes

// (T 2^32 + L) 2^e rounded half up to FP64, |T| < 2^46, |L| < 2^50, by
// assembling the bits; overflow gives an infinity
__device__ __forceinline__ double sum_value(long long T, long long L, int e) {
  unsigned l, h0, h1, l0, l1;
  split64(L, l, l1);
  split64(T + (long long)(int)l1, h0, h1);
  const unsigned sign = h1 & 0x80000000u;
  if (sign)
    asm("sub.cc.u32 %0, 0, %0;\n\tsubc.cc.u32 %1, 0, %1;\n\tsubc.u32 %2, 0, %2;" : "+r"(l), "+r"(h0), "+r"(h1));
  if ((h0 | h1) == 0u) {
    if (l == 0u) return 0.0;
    h0 = l;
    l = 0u;
    e -= 32;
  }
  const bool one = h1 == 0u;                           // the top word is h0
  const int lz = one ? __clz(h0) : __clz(h1);
  const unsigned w2 = one ? h0 : h1, w1 = one ? l : h0, w0 = one ? 0u : l;
  l1 = __funnelshift_l(w1, w2, lz);                    // bit 31 of l1 set
  l0 = __funnelshift_l(w0, w1, lz);
  int E = 1023 + (one ? 63 : 95) - lz + e;
  if (E <= 0) {                                        // subnormal: 12 - E bits go; a carry makes 2^-1022
    const int s = 11 - E;
    const unsigned long long m = s > 63 ? 0ull : (unsigned long long)join64(l0, l1) >> s;
    return __longlong_as_double((long long)(((m + 1ull) >> 1) | ((unsigned long long)sign << 32)));
  }
  unsigned cy;
  asm("add.cc.u32 %0, %0, 1024;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, 0, 0;" : "+r"(l0), "+r"(l1), "=r"(cy));
  if (cy) {                                            // rounded up to a power of two
    l1 = 0x80000000u;
    l0 = 0u;
    E += 1;
  }
  if (E >= 2047) return __hiloint2double((int)(sign | 0x7ff00000u), 0);
  return __hiloint2double((int)(sign | ((unsigned)E << 20) | ((l1 >> 11) & 0xfffffu)),
                          (int)__funnelshift_r(l0, l1, 11));
}

// x (of a line whose largest exponent field is e, at least 1) as a 60-bit integer,
// x 2^(1082 - e) rounded (truncation towards zero would bias the low modes);
// subnormals have the exponent of field 1 and no leading bit
__device__ __forceinline__ long long line_int(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)((hi >> 20) & 0x7ffu);
  const int s = e - max(ex, 1);
  const unsigned mh = (hi & 0xfffffu) | (ex == 0 ? 0u : 0x100000u);
  const unsigned long long m = (unsigned long long)join64(lo << 8, __funnelshift_l(lo, mh, 8));
  const long long v = s > 62 ? 0ll : (long long)(((m >> s) + 1ull) >> 1);
  return (int)hi < 0 ? -v : v;
}

// Two integers as 16 bytes: word w holds digits 2w and 2w + 1 (digit 0 the top
// byte) of both, interleaved, with the bias 128 of a balanced digit in place.
__device__ __forceinline__ uint4 pack_digits(long long a, long long b) {
  const unsigned long long bias = 0x8080808080808080ull;
  const unsigned long long ua = (unsigned long long)a + bias, ub = (unsigned long long)b + bias;
  const unsigned la = (unsigned)ua, ha = (unsigned)(ua >> 32), lb = (unsigned)ub, hb = (unsigned)(ub >> 32);
  return make_uint4(__byte_perm(ha, hb, 0x6273), __byte_perm(ha, hb, 0x4051), __byte_perm(la, lb, 0x6273),
                    __byte_perm(la, lb, 0x4051));
}

// digits 2w, 2w + 1 of both integers as FP16 pairs: 0x6400 | byte is 1024 + byte
__device__ __forceinline__ void unpack_digits(unsigned w, unsigned& d0, unsigned& d1) {
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));   // 1152
  const unsigned r0 = __byte_perm(w, 0x64646464u, 0x4140), r1 = __byte_perm(w, 0x64646464u, 0x4342);
  const __half2 h0 = __hsub2(*reinterpret_cast<const __half2*>(&r0), off);
  const __half2 h1 = __hsub2(*reinterpret_cast<const __half2*>(&r1), off);
  d0 = *reinterpret_cast<const unsigned*>(&h0);
  d1 = *reinterpret_cast<const unsigned*>(&h1);
}

// The eight sums of digit products (integers in FP32, at most 2^24) as
// R = T 2^32 + L.  A float-to-int conversion issues to the XU pipe, so the
// integers are read from the bits of f + 1.5 2^23, exact up to 2^22; larger
// sums, which only crafted digits reach, are split first.
__device__ __forceinline__ void sum_digits(const float (&f)[8], long long& T, long long& L) {
  const float magic = 12582912.f;
  float m = 0.f;
#pragma unroll
  for (int d = 0; d < 8; ++d) m = fmaxf(m, fabsf(f[d]));
  if (m <= 4194304.f) {
    // pairs in 32 bits, the offsets 0x4B400000 of both taken off together
    constexpr unsigned off = 0x4B400000u * 257u;
    unsigned b[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) b[d] = (unsigned)__float_as_int(__fadd_rn(f[d], magic));
    const int p0 = (int)(b[0] * 256u + b[1] - off), p1 = (int)(b[2] * 256u + b[3] - off);
    const int p2 = (int)(b[4] * 256u + b[5] - off), p3 = (int)(b[6] * 256u + b[7] - off);
    T = add64(join64((unsigned)p0 << 16, (unsigned)(p0 >> 16)), join64((unsigned)p1, (unsigned)(p1 >> 31)));
    L = add64(join64((unsigned)p2 << 16, (unsigned)(p2 >> 16)), join64((unsigned)p3, (unsigned)(p3 >> 31)));
  } else {
    int w[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) w[d] = __float2int_rn(f[d]);
    T = (long long)(w[0] * 256 + w[1]) * 65536 + ((long long)w[2] * 256 + w[3]);
    L = (long long)w[4] * 16777216 + ((long long)w[5] * 65536 + ((long long)w[6] * 256 + w[7]));
  }
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Mode tiles of 16: tiles [0, T) hold k = 2i + 1, [T, 3T/2) k = 4i + 2,
// [3T/2, 2T) k = 4i + 4 (its last row, k = N, is empty), T = N / 32.
struct MmaTile {
  int k0, kstep;     // row r is mode k0 + r kstep
  int pair0;         // first digit pair of the class in a line's packed buffer
  int nks;           // steps of 16 terms
  long long frag;    // first fragment (uint4 index) of the tile in the table
};
__host__ __device__ __forceinline__ MmaTile mma_tile(int n, int t) {
  const int T = n >> 5;
  MmaTile m;
  if (t < T) {
    m = MmaTile{32 * t + 1, 2, 0, n >> 5, (long long)t * (n >> 5) * 128};
  } else {
    const int u = t - T, h = T >> 1;
    m.kstep = 4;
    m.nks = n >> 6;
    m.frag = ((long long)T * (n >> 5) + (long long)u * (n >> 6)) * 128;
    if (u < h) {
      m.k0 = 64 * u + 2;
      m.pair0 = n >> 2;
    } else {
      m.k0 = 64 * (u - h) + 4;
      m.pair0 = 3 * (n >> 3);
    }
  }
  return m;
}
__host__ __device__ __forceinline__ long long mma_frag_count(int n) {   // uint4 entries of the table
  const long long T = n >> 5;
  return (T * (n >> 5) + T * (n >> 6)) * 128;
}

// The matrix in fragment order: entry [tile][step][q][lane] is the digit pair
// of terms j = 16 step + 2 (lane % 4) + 8 (q / 2) + {1, 2}, row lane / 4 + 8 (q % 2).
// sq[i] = round(2^62 sin(pi i / N)), i = 0..N (exact to the last bit or two).
__global__ void k_mma_table(int n, const long long* __restrict__ sq, uint4* __restrict__ frag) {
  const long long tot = mma_frag_count(n);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const int lane = (int)(e & 31), q = (int)((e >> 5) & 3);
    const long long ts = e >> 7;                    // tile and step
    const int T = n >> 5;
    const long long odd = (long long)T * (n >> 5);
    const int t = ts < odd ? (int)(ts / (n >> 5)) : T + (int)((ts - odd) / (n >> 6));
    const MmaTile m = mma_tile(n, t);
    const int step = (int)(ts - m.frag / 128);
    const int k = m.k0 + m.kstep * ((lane >> 2) + 8 * (q & 1));
    long long v[2];
    for (int i = 0; i < 2; ++i) {
      const int j = 16 * step + 2 * (lane & 3) + 8 * (q >> 1) + i + 1;
      const int a = (int)(((long long)k * j) % (2 * n));
      v[i] = a <= n ? sq[a] : -sq[a - n];
    }
    frag[e] = pack_digits(v[0], v[1]);
  }
}

// Layout of a CTA's shared memory: NL lines of n/2 + 4 digit pairs, NL lines
// of n + 4 FP64 (or int64) values, value j at j - 1 (the paddings spread a
// fragment's rows over the banks), NL exponents.
template <int LOGN, int W>
struct Mma {
  static constexpr int N = 1 << LOGN, NL = 8, THREADS = 32 * W;
  static constexpr int PR = N + 4, PP = N / 2 + 4;
  static constexpr int VALS = N * NL / THREADS;        // elements per thread
  static constexpr bool BIG = N > 256;                 // K > 128: the sums are emptied every 128 terms
  static constexpr size_t SMEM = (size_t)NL * (PR * 8 + PP * 16) + NL * sizeof(int);
};

// Element i of this thread: contiguous lines by a warp per line, strided ones
// with the CTA's adjacent lines side by side.
template <int LOGN, int W>
__device__ __forceinline__ void mma_coord(bool contig, int i, int& q, int& j) {
  using M = Mma<LOGN, W>;
  constexpr int PER = M::N / 32;
  if (contig) {
    q = (threadIdx.x >> 5) + W * (i / PER);
    j = (threadIdx.x & 31) + 32 * (i % PER);
  } else {
    q = threadIdx.x % M::NL;
    j = threadIdx.x / M::NL + (M::THREADS / M::NL) * i;
  }
}

// The lines' values x (as mma_coord deals them) as 60-bit integers in raw,
// their exponents in sexp (1 on entry), then the foldings as digit pairs.
template <int LOGN, int W>
__device__ __forceinline__ void mma_fold(double (&x)[Mma<LOGN, W>::VALS], bool contig, double* raw, uint4* pk,
                                         int* sexp) {
  using M = Mma<LOGN, W>;
  constexpr int n = M::N, NL = M::NL, VALS = M::VALS, PER = n / 32, pr = M::PR, pp = M::PP;
  if (contig) {
#pragma unroll
    for (int l = 0; l < VALS / PER; ++l) {
      unsigned mx = 0u;
#pragma unroll
      for (int i = 0; i < PER; ++i) mx = max(mx, (unsigned)__double2hiint(x[l * PER + i]) & 0x7fffffffu);
      mx = __reduce_max_sync(0xffffffffu, mx);
      if ((threadIdx.x & 31) == 0) sexp[(threadIdx.x >> 5) + W * l] = max((int)(mx >> 20), 1);
    }
    __syncwarp();                                      // a warp reads its own lines' exponents
  } else {
    unsigned mx = 0u;
#pragma unroll
    for (int i = 0; i < VALS; ++i) mx = max(mx, (unsigned)__double2hiint(x[i]) & 0x7fffffffu);
#pragma unroll
    for (int o = NL; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) < NL) atomicMax(sexp + threadIdx.x % NL, (int)(mx >> 20));
    __syncthreads();
  }
  long long* xi = reinterpret_cast<long long*>(raw);
#pragma unroll
  for (int i = 0; i < VALS; ++i) {
    int q, j;
    mma_coord<LOGN, W>(contig, i, q, j);
    if (j > 0) xi[q * pr + j - 1] = line_int(x[i], sexp[q]);
  }
  __syncthreads();
  constexpr int half = n / 2, quart = n / 4, eighth = n / 8;
#pragma unroll 4
  for (int t = threadIdx.x; t < NL * half; t += M::THREADS) {
    const int q = t / half, s = t % half;
    const long long* v = xi + q * pr - 1;              // v[j] is element j
    long long r0, r1;
    if (s < quart) {
      const int j = 2 * s + 1;
      r0 = v[j] + v[n - j];
      r1 = v[j + 1] + (j + 1 == half ? 0ll : v[n - j - 1]);
    } else {
      const bool minus = s >= quart + eighth;
      const int j = 2 * (s - (minus ? quart + eighth : quart)) + 1;
      const long long a0 = v[j] - v[n - j], b0 = v[half - j] - v[half + j];
      const long long a1 = v[j + 1] - v[n - j - 1], b1 = v[half - j - 1] - v[half + j + 1];
      r0 = minus ? a0 - b0 : a0 + b0;
      // at j + 1 = N/4 the two terms are one
      r1 = minus ? (j + 1 == quart ? 0ll : a1 - b1) : (j + 1 == quart ? a1 : a1 + b1);
    }
    pk[q * pp + s] = pack_digits(r0, r1);
  }
  __syncthreads();
}

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// All mode tiles t = t0, t0 + ts, ... of the CTA's lines: X_k = sum_j
// x_j sin(pi k j / N) into raw; with `scale` (the first half of the fused
// pass) times the spectral scale, into raw of every CTA of the cluster.  No
// raw is written before every CTA of the cluster has read its lines.
template <int LOGN, int W>
__device__ __forceinline__ void mma_modes(const PassArgs& A, int t0, int ts, const uint4* __restrict__ frag,
                                          const uint4* pk, const int* sexp, double* raw, int a, int b0, bool scale) {
  using M = Mma<LOGN, W>;
  constexpr int n = M::N, pr = M::PR, pp = M::PP;
  constexpr bool BIG = M::BIG;
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int peers = scale ? (int)gridDim.z : 1;        // the cluster is the grid's z extent
  // spectral scale of accumulator v of a tile (1 off the grid)
  auto scale_at = [&](const MmaTile& m, int v) {
    const int b = b0 + 2 * c + (v & 1), k = m.k0 + m.kstep * (g + 8 * (v >> 1)), m1 = n - 1;
    if (b >= n || k >= n) return 1.0;
    return __ldg(A.scale64 + (A.d == 2 ? (k - 1) * m1 + b - 1 : ((k - 1) * m1 + a - 1) * m1 + b - 1));
  };
  constexpr bool AHEAD = LOGN > 9;
  bool waited = false;
  for (int t = t0; t < n / 16; t += ts) {
    const MmaTile m = mma_tile(n, t);
    const uint4* fr = frag + m.frag + lane;
    const uint4* pb = pk + g * pp + m.pair0 + c;
    float acc[8][4];
    long long sT[BIG ? 4 : 1], sL[BIG ? 4 : 1];
#pragma unroll
    for (int d = 0; d < 8; ++d)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[d][v] = 0.f;
    if (BIG)
#pragma unroll
      for (int v = 0; v < 4; ++v) sT[v] = sL[v] = 0ll;
    // N = 1024: the tile's scales before its products, which hide their latency (one
    // CTA per SM does not; smaller N have no registers left for them).  Two operators'
    // grids exceed L2: general right-hand side 956 -> 930 us, evaluation 936 -> 914,
    // with mma_prefetch 916 and 897 (by FFT 919 and 908)
    double scl[AHEAD ? 4 : 1];
    if (AHEAD && scale)
#pragma unroll
      for (int v = 0; v < 4; ++v) scl[v] = scale_at(m, v);
    uint4 fa[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) fa[q] = __ldg(fr + 32 * q);
#pragma unroll 1
    for (int ks = 0; ks < m.nks; ++ks) {
      unsigned ad[8][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        unpack_digits(fa[q].x, ad[0][q], ad[1][q]);
        unpack_digits(fa[q].y, ad[2][q], ad[3][q]);
        unpack_digits(fa[q].z, ad[4][q], ad[5][q]);
        unpack_digits(fa[q].w, ad[6][q], ad[7][q]);
      }
      if (ks + 1 < m.nks) {
        fr += 128;
#pragma unroll
        for (int q = 0; q < 4; ++q) fa[q] = __ldg(fr + 32 * q);
      }
      const uint4 p0 = pb[0], p1 = pb[4];
      pb += 8;
      unsigned bd[8][2];
      unpack_digits(p0.x, bd[0][0], bd[1][0]);
      unpack_digits(p0.y, bd[2][0], bd[3][0]);
      unpack_digits(p0.z, bd[4][0], bd[5][0]);
      unpack_digits(p0.w, bd[6][0], bd[7][0]);
      unpack_digits(p1.x, bd[0][1], bd[1][1]);
      unpack_digits(p1.y, bd[2][1], bd[3][1]);
      unpack_digits(p1.z, bd[4][1], bd[5][1]);
      unpack_digits(p1.w, bd[6][1], bd[7][1]);
      // by rows of digit i: neighbouring products go to different sums
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8 - i; ++j) mma_f16(acc[i + j], ad[i], bd[j]);
      if (BIG && (ks & 7) == 7) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          float f[8];
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            f[d] = acc[d][v];
            acc[d][v] = 0.f;
          }
          long long T, L;
          sum_digits(f, T, L);
          sT[v] += T;
          sL[v] += L;
        }
      }
    }
    if (!waited) {
      cluster_wait();
      waited = true;
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int q = 2 * c + (v & 1);
      const int k = m.k0 + m.kstep * (g + 8 * (v >> 1));
      if (k >= n) continue;
      long long T, L;
      if (BIG) {
        T = sT[v];
        L = sL[v];
      } else {
        float f[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) f[d] = acc[d][v];
        sum_digits(f, T, L);
      }
      const int e = sexp[q];
      // units: digits 7 of both factors 2^56, the matrix 2^62, the line 2^(1082 - e)
      double r = sum_value(T, L, e - 1088);
      if (e == 0x7ff) r = __longlong_as_double(0x7ff8000000000000LL);   // a non-finite line
      if (scale) r *= AHEAD ? scl[AHEAD ? v : 0] : scale_at(m, v);
      if (peers == 1) {
        raw[q * pr + k - 1] = r;
      } else {
        for (int z = 0; z < peers; ++z) cluster.map_shared_rank(raw, z)[q * pr + k - 1] = r;
      }
    }
  }
  if (!waited) cluster_wait();
}

// 2D, N = 1024: the digit table (2.2 MB) and the CTA's spectral scales on their way
// into L2.  All CTAs walk the table in step, so where other grids have pushed it out,
// it is else a chain of misses: operator on a problem not used just before 442 ->
// 420 us (by FFT 428).  At 512^2 (0.6 MB) the requests cost more than they bring (86.0
// against 85.3 us).
template <int LOGN, int W>
__device__ __forceinline__ void mma_prefetch(const PassArgs& A, const uint4* frag, int b0) {
  using M = Mma<LOGN, W>;
  constexpr int n = M::N;
  auto fetch = [](const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); };
  const int cta = blockIdx.z * gridDim.x + blockIdx.x, t = cta * M::THREADS + threadIdx.x;
  for (int k = t; k < (int)(mma_frag_count(n) / 8); k += gridDim.x * gridDim.z * M::THREADS) fetch(frag + 8 * (long long)k);
  if (A.fused)
    for (int k = threadIdx.x; k < n - 1; k += M::THREADS) fetch(A.scale64 + (long long)k * (n - 1) + b0 - 1);
}

// One pass over the 8 lines b0.. of family a: W warps; the gridDim.z CTAs of a
// cluster all read the lines and share their modes.
template <int LOGN, int W>
__global__ void __launch_bounds__(32 * W, LOGN > 9 ? 1 : W == 8 ? 2 : 4) k_dst_mma(PassArgs A) {
  using M = Mma<LOGN, W>;
  constexpr int n = M::N, NL = M::NL, VALS = M::VALS, pr = M::PR;
  extern __shared__ __align__(16) unsigned char smraw[];
  uint4* pk = reinterpret_cast<uint4*>(smraw);
  double* raw = reinterpret_cast<double*>(pk + NL * M::PP);
  int* sexp = reinterpret_cast<int*>(raw + NL * pr);
  const uint4* frag = static_cast<const uint4*>(A.frag);
  const int a = blockIdx.y + 1, b0 = 1 + NL * blockIdx.x;
  const int sb = (int)A.sb, es = (int)A.es, off0 = a * (int)A.sa + b0 * sb;   // 32-bit: at most 1025^3 nodes
  const bool contig = es == 1;
  if (threadIdx.x < NL) sexp[threadIdx.x] = 1;
  if (LOGN > 9 && A.d == 2) mma_prefetch<LOGN, W>(A, frag, b0);
  double x[VALS];
  {
    const double* src = static_cast<const double*>(A.src) + off0;
#pragma unroll
    for (int i = 0; i < VALS; ++i) {
      int q, j;
      mma_coord<LOGN, W>(contig, i, q, j);
      x[i] = (j > 0 && b0 + q < n) ? src[q * sb + j * es] : 0.0;
    }
  }
  __syncthreads();
  mma_fold<LOGN, W>(x, contig, raw, pk, sexp);
  cluster_arrive();
  const int t0 = (threadIdx.x >> 5) * gridDim.z + blockIdx.z, ts = W * gridDim.z;
  mma_modes<LOGN, W>(A, t0, ts, frag, pk, sexp, raw, a, b0, A.fused != 0);
  if (A.fused) {
    cluster_arrive();
    cluster_wait();                                    // every mode of the lines is in raw
#pragma unroll
    for (int i = 0; i < VALS; ++i) {
      int q, j;
      mma_coord<LOGN, W>(true, i, q, j);
      x[i] = j > 0 ? raw[q * pr + j - 1] : 0.0;
    }
    __syncthreads();
    mma_fold<LOGN, W>(x, true, raw, pk, sexp);
    cluster_arrive();
    mma_modes<LOGN, W>(A, t0, ts, frag, pk, sexp, raw, a, b0, false);
  }
  __syncthreads();
  double* dst = static_cast<double*>(A.dst) + off0;
  if (gridDim.z == 1) {
#pragma unroll
    for (int i = 0; i < VALS; ++i) {
      int q, j;
      mma_coord<LOGN, W>(contig, i, q, j);
      if (j > 0 && b0 + q < n) dst[q * sb + j * es] = raw[q * pr + j - 1];
    }
  } else {
    // this CTA's modes only
    for (int tt = blockIdx.z; tt < n / 16; tt += gridDim.z) {
      const MmaTile m = mma_tile(n, tt);
      for (int t = threadIdx.x; t < NL * 16; t += M::THREADS) {
        const int r = contig ? t & 15 : t / NL;
        const int q = contig ? t >> 4 : t % NL;
        const int k = m.k0 + m.kstep * r;
        if (k < n && b0 + q < n) dst[q * sb + k * es] = raw[q * pr + k - 1];
      }
    }
  }
}

}  // namespace
}  // namespace kfbi

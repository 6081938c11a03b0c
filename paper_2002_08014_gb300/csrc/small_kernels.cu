// The d x k and k x k kernels around the fused power step:
//   reduce     Y_i = (1/s_i) sum of the step kernel's per-CTA partials (fixed order)
//   align      sign-fixing (eq. (4)) or orthogonal Procrustes (eq. (3)) matrices
//   aggregate  Y = sum_i p_i Y_i D_i (Alg. 1 aggregation)
//   ritz       Rayleigh-Ritz on span(Z): ordered basis and sigma_j = sqrt(n lambda_j)
//   split      FP32 rows -> hi / lo BF16 planes (load time)
//   rho        residual error of Def. 3 per partition (traced solves)
// (the orthonormalisation is in cholqr2.cu).
// Precision, by default: the d-sized work (averaging) and the k x k Jacobi SVD /
// eigen-solves are FP32; the Ritz matrix H is accumulated in FP64, and the sign-fix
// inner products that decide D_i are wherever an FP32 sum's error bound leaves the
// sign open.  GB300's FP64 pipe is a small fraction of its FP32 pipe, and these k x k
// steps are serial latency on every round.  With LP_FLAG_KXK_FP64 the Procrustes SVD
// and the Ritz eigen-solve are FP64 too.
#include <algorithm>
#include <cfloat>
#include <mutex>
#include <unordered_set>

#include <cuda_bf16.h>

#include "inv_sqrt.cuh"
#include "lp_internal.cuh"

namespace lp {
namespace {

constexpr int kT = 256;

// ---------------------------------------------------------------- pack / unpack
// FP32 rows -> two BF16 planes: hi = RNE(a), lo = RNE(a - hi).  a - hi is exact
// in FP32, so hi + lo matches a to within half an ulp of lo (<= 2^-17 |a|).
// Bound by HBM (4 bytes read, 4 written per element).  One launch takes up to
// kSplitParts partitions, so that a load of many small ones has no launch tails;
// a thread converts eight columns of a row (two 16-byte loads, one 16-byte store
// per plane) and has two such groups in flight.  Rows that are not 16-byte
// aligned, and a row's last columns, are read one by one.  Measured, 64 partitions
// of 2,048 x 1,024: 732 us (64 launches, an element per thread) -> 158 us, 6.8 TB/s.
__device__ __forceinline__ void split8(const float* __restrict__ src, int64_t src_ld, bool vec, int64_t row, int c, int d,
                                       float (&v)[8]) {
  const float* p = src + row * src_ld + c;
  if (vec && c + 8 <= d) {
    const float4 x = reinterpret_cast<const float4*>(p)[0], y = reinterpret_cast<const float4*>(p)[1];
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = c + q < d ? p[q] : 0.f;
  }
}

__global__ void __launch_bounds__(kT) split_planes_kernel(const __grid_constant__ SplitParts parts, int64_t src_ld,
                                                          int d, uint16_t* __restrict__ hi,
                                                          uint16_t* __restrict__ lo, int ld8) {
  const int64_t total = parts.row0[parts.n] * ld8;
  const int64_t step = int64_t(gridDim.x) * kT;
  int part = 0;
  for (int64_t e0 = blockIdx.x * int64_t(kT) + threadIdx.x; e0 < total; e0 += 2 * step) {
    float v[2][8];
    int64_t at[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int64_t e = e0 + x * step;
      at[x] = -1;
      if (e >= total) continue;
      int64_t r;
      int c;
      if (total < (int64_t(1) << 31)) {
        r = static_cast<uint32_t>(e) / static_cast<uint32_t>(ld8);
        c = static_cast<int>(static_cast<uint32_t>(e) - static_cast<uint32_t>(r) * ld8);
      } else {
        r = e / ld8;
        c = static_cast<int>(e - r * ld8);
      }
      while (r >= parts.row0[part + 1]) ++part;  // a thread's rows ascend
      const float* src = parts.src[part];
      const bool vec = ((reinterpret_cast<uintptr_t>(src) | static_cast<uintptr_t>(src_ld * 4)) & 15) == 0;
      split8(src, src_ld, vec, r - parts.row0[part], 8 * c, d, v[x]);
      at[x] = e;
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      if (at[x] < 0) continue;
      uint32_t h[4], l[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float a0 = v[x][2 * q], a1 = v[x][2 * q + 1];
        const __nv_bfloat16 h0 = __float2bfloat16_rn(a0), h1 = __float2bfloat16_rn(a1);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(a0 - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(a1 - __bfloat162float(h1));
        h[q] = __bfloat16_as_ushort(h0) | (static_cast<uint32_t>(__bfloat16_as_ushort(h1)) << 16);
        l[q] = __bfloat16_as_ushort(l0) | (static_cast<uint32_t>(__bfloat16_as_ushort(l1)) << 16);
      }
      reinterpret_cast<uint4*>(hi)[at[x]] = make_uint4(h[0], h[1], h[2], h[3]);
      reinterpret_cast<uint4*>(lo)[at[x]] = make_uint4(l[0], l[1], l[2], l[3]);
    }
  }
}

// FP64 rows of k -> FP32 rows of K, zero beyond k; a thread converts four columns
// of a row (K is a multiple of four).  `clear` (may be nullptr): a status word to
// zero, for kernels later on the stream.
__global__ void __launch_bounds__(kT) pack_kernel(const double* __restrict__ src, float* __restrict__ dst, int64_t rows,
                                                  int k, int K, int* clear) {
  if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
  const int KQ = K / 4;
  const bool vec = k % 4 == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  const int64_t total = rows * KQ;
  for (int64_t e = blockIdx.x * int64_t(kT) + threadIdx.x; e < total; e += int64_t(gridDim.x) * kT) {
    const int64_t row = e / KQ;
    const int j = 4 * static_cast<int>(e - row * KQ);
    const double* p = src + row * k + j;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec && j + 4 <= k) {
      const double2 x = reinterpret_cast<const double2*>(p)[0], y = reinterpret_cast<const double2*>(p)[1];
      v = make_float4(static_cast<float>(x.x), static_cast<float>(x.y), static_cast<float>(y.x), static_cast<float>(y.y));
    } else {
      if (j < k) v.x = static_cast<float>(p[0]);
      if (j + 1 < k) v.y = static_cast<float>(p[1]);
      if (j + 2 < k) v.z = static_cast<float>(p[2]);
      if (j + 3 < k) v.w = static_cast<float>(p[3]);
    }
    reinterpret_cast<float4*>(dst)[e] = v;
  }
}
__global__ void to_float_kernel(const double* __restrict__ src, float* __restrict__ dst, int n) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) dst[e] = static_cast<float>(src[e]);
}
// The inverse: FP32 rows of K -> FP64 rows of k.
__device__ __forceinline__ void store_f64(double* __restrict__ row, int j, int k, bool vec, float4 v) {
  if (vec && j + 4 <= k) {
    reinterpret_cast<double2*>(row + j)[0] = make_double2(v.x, v.y);
    reinterpret_cast<double2*>(row + j)[1] = make_double2(v.z, v.w);
  } else {
    if (j < k) row[j] = v.x;
    if (j + 1 < k) row[j + 1] = v.y;
    if (j + 2 < k) row[j + 2] = v.z;
    if (j + 3 < k) row[j + 3] = v.w;
  }
}
__global__ void __launch_bounds__(kT) unpack_kernel(const float* __restrict__ src, double* __restrict__ dst,
                                                    int64_t rows, int k, int K) {
  const int KQ = K / 4;
  const bool vec = k % 4 == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
  const int64_t total = rows * KQ;
  for (int64_t e = blockIdx.x * int64_t(kT) + threadIdx.x; e < total; e += int64_t(gridDim.x) * kT) {
    const int64_t row = e / KQ;
    const int j = 4 * static_cast<int>(e - row * KQ);
    if (j < k) store_f64(dst + row * k, j, k, vec, reinterpret_cast<const float4*>(src)[e]);
  }
}

// ---------------------------------------------------------------- reduce
// G adjacent threads share one float4 of Y_i: thread g of the group sums slots
// sb + g, sb + g + G, ... in order (four loads in flight), then the group adds
// its G partials by an xor butterfly.  The order is fixed for a given G, so
// results are reproducible; G > 1 only when partitions have many slots (small
// problems spread over many CTAs), where it cuts the chain of dependent loads.
// OUT64: the sums go to the caller's FP64 rows of k (the single power step, which
// needs no FP32 copy: 128 blocks of 2,048 x 32, 18 + 25 us as two kernels), and the
// first thread hands the status word to host memory.
template <int G, bool OUT64>
__global__ void reduce_kernel(const float* __restrict__ P, const int* __restrict__ slot_begin,
                              const float* __restrict__ scale, int d, int K, float* __restrict__ Y,
                              double* __restrict__ Yd, int k, const int* status, int* status_host) {
  const int i = blockIdx.y;
  after_previous();
  before_next();
  if (OUT64 && status_host && blockIdx.x == 0 && i == 0 && threadIdx.x == 0) *status_host = *status;
  const int64_t n4 = int64_t(d) * K / 4;
  const int g = threadIdx.x % G;
  const int64_t e = blockIdx.x * int64_t(blockDim.x / G) + threadIdx.x / G;
  const bool live = e < n4;
  if (G == 1 && !live) return;
  const int sb = slot_begin[i], se = slot_begin[i + 1];
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live) {
    int s = sb + g;
    for (; s + 3 * G < se; s += 4 * G) {
      float4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = reinterpret_cast<const float4*>(P + int64_t(s + q * G) * d * K)[e];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc.x += v[q].x; acc.y += v[q].y; acc.z += v[q].z; acc.w += v[q].w;
      }
    }
    for (; s < se; s += G) {
      const float4 v = reinterpret_cast<const float4*>(P + int64_t(s) * d * K)[e];
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
  }
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
    acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
  }
  if (!live || g != 0) return;
  const float sc = scale[i];
  acc.x *= sc; acc.y *= sc; acc.z *= sc; acc.w *= sc;
  if constexpr (OUT64) {
    const int KQ = K / 4, row = static_cast<int>(e / KQ), j = 4 * static_cast<int>(e - int64_t(row) * KQ);
    const bool vec = k % 4 == 0 && (reinterpret_cast<uintptr_t>(Yd) & 15) == 0;
    if (j < k) store_f64(Yd + (int64_t(i) * d + row) * k, j, k, vec, acc);
  } else {
    reinterpret_cast<float4*>(Y + int64_t(i) * d * K)[e] = acc;
  }
}

// ---------------------------------------------------------------- k x k helpers
__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Thresholds of the Jacobi sweeps per precision: a pair (p, q) is rotated while
// |c_p . c_q| > tol ||c_p|| ||c_q|| (tol a few units of the type's rounding
// error times k, so the last sweep only sees rounding noise below it); `tiny`
// skips pairs whose product underflows; beyond `huge` t = 1 / (2 |zeta|) avoids
// squaring zeta.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float inv_root(float x) { return inv_sqrt(x); }
__device__ __forceinline__ double inv_root(double x) { return 1.0 / sqrt(x); }
template <typename T> struct JacobiLimits;
template <> struct JacobiLimits<float> {
  static constexpr float tol = 1e-6f, tiny = 1e-35f, huge = 1e15f;
};
template <> struct JacobiLimits<double> {
  static constexpr double tol = 1e-13, tiny = 1e-300, huge = 1e150;
};

// One-sided (Hestenes) Jacobi on the k x k matrix C (stride ks, in shared memory),
// accumulating the rotations in V, in precision T: on return C's columns are
// mutually orthogonal, C_in V = C_out, so C_in = U Sigma V^T with
// sigma_j = ||C_out[:, j]|| and U[:, j] = C_out[:, j] / sigma_j.  FP32 by
// default because GB300's FP64 pipe is a small fraction of its FP32 pipe and
// these k x k problems sit on serial critical paths (the aligners and Ritz
// values stay within 1e-7 of FP64 factorisations on the FP32 workload's
// spectrum); FP64 under LP_FLAG_KXK_FP64.
//
// All kT threads of the CTA call it.  A sweep visits every column pair once in
// the round-robin (circle) order: with np = k rounded up to even (the extra
// column a dummy whose pairs are skipped), step s pairs column np - 1 with s and
// (s + j) mod (np - 1) with (s - j) mod (np - 1) for j = 1 .. np/2 - 1, which
// makes each step a set of disjoint pairs and each sweep np - 1 steps.  Pair
// slot j of a step belongs to half-warp j; its 16 lanes hold rows h and h + 16
// of the two columns, sum the three inner products over the half-warp and
// rotate their rows.  One barrier per step; the sweeps stop when a whole sweep
// rotated nothing.  Returns false if the sweep limit was hit.
// ks = jacobi_stride(K), one past K: a half-warp reads 16 rows of one column, which
// at a stride of 32 words would all lie in one bank (OPT align, 20 blocks of 362 x 24:
// 212 -> 90 us with it, the pair's rows read once and the rotation's root as inv_sqrt;
// 64 of 1,024 x 16: 82 -> 50).  What is left is the chain of a step, ~750 cycles: the
// four shuffles, two divisions and two roots, and the barrier.
__host__ __device__ constexpr int jacobi_stride(int K) { return K + 1; }
template <typename T>
__device__ bool cta_jacobi(T* C, T* V, int k, int K) {
  const int ks = jacobi_stride(K);
  using L = JacobiLimits<T>;
  const int t = threadIdx.x;
  const int slot = t >> 4, h = t & 15;
  const int np = k + (k & 1);
  for (int e = t; e < K * K; e += kT) V[e / K * ks + e % K] = (e / K == e % K) ? T(1) : T(0);
  __syncthreads();
  for (int sweep = 0; sweep < 40; ++sweep) {
    int rotated = 0;
    for (int s = 0; s < np - 1; ++s) {
      int p = 0, q = 0;
      bool live = slot < np / 2;
      if (live) {
        p = s + (slot == 0 ? 0 : slot);
        if (p >= np - 1) p -= np - 1;
        q = slot == 0 ? np - 1 : s - slot;
        if (q < 0) q += np - 1;
        live = p < k && q < k;
      }
      // rows h and h + 16 of the pair, read once for the products and the rotation
      const bool r0 = live && h < k, r1 = live && h + 16 < k;
      T *c0 = C + h * ks, *c1 = c0 + 16 * ks;
      const T p0 = r0 ? c0[p] : T(0), q0 = r0 ? c0[q] : T(0);
      const T p1 = r1 ? c1[p] : T(0), q1 = r1 ? c1[q] : T(0);
      T a = 0, b = 0, g = 0;
      if (__any_sync(0xffffffffu, live)) {  // a warp without a pair skips the sums (FP64: its pipe is the bound)
        a = mul_rn(p0, p0);
        b = mul_rn(q0, q0);
        g = mul_rn(p0, q0);
        if (k > 16) {
          a = fma(p1, p1, a);
          b = fma(q1, q1, b);
          g = fma(p1, q1, g);
        }
        // every lane takes part in the shuffles; offsets below 16 stay in the half-warp
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
          a += __shfl_xor_sync(0xffffffffu, a, o);
          b += __shfl_xor_sync(0xffffffffu, b, o);
          g += __shfl_xor_sync(0xffffffffu, g, o);
        }
      }
      if (live && fabs(g) > L::tol * sqrt(a * b) && fabs(g) > L::tiny) {
        rotated = 1;
        // zeta = (b - a) / 2g, t = sgn(zeta) / (|zeta| + sqrt(1 + zeta^2)), c = 1 / sqrt(1 + t^2)
        const T zeta = (b - a) / (T(2) * g);
        const T az = fabs(zeta);
        const T tn = (zeta >= T(0) ? T(1) : T(-1)) / (az > L::huge ? T(2) * az : az + sqrt(fma(zeta, zeta, T(1))));
        const T c = inv_root(fma(tn, tn, T(1)));
        const T sn = c * tn;
        // a rotated pair of values: (c x - s y, s x + c y), one product of each rounded first
        auto rot = [&](T x, T y, T& lo, T& hi) {
          lo = fma(c, x, -mul_rn(sn, y));
          hi = fma(sn, x, mul_rn(c, y));
        };
        T *v0 = V + h * ks, *v1 = v0 + 16 * ks;
        if (r0) {
          const T vp = v0[p], vq = v0[q];
          rot(p0, q0, c0[p], c0[q]);
          rot(vp, vq, v0[p], v0[q]);
        }
        if (r1) {
          const T vp = v1[p], vq = v1[q];
          rot(p1, q1, c1[p], c1[q]);
          rot(vp, vq, v1[p], v1[q]);
        }
      }
      __syncthreads();
    }
    if (!__syncthreads_or(rotated)) return true;
  }
  return false;
}

// The orthogonal Procrustes factor O = U V^T of eq. (3) from a finished one-sided
// Jacobi (C holds U Sigma, V the rotations): U's columns are normalised in
// place, then O is formed entry by entry into Gi (K x K, zero beyond k).  A
// column with no norm leaves O short of orthogonal and sets ST_JACOBI.  All
// threads call it; `inv` holds K values of scratch.
template <typename T>
__device__ void procrustes_factor(T* C, const T* V, T* inv, int k, int K, float* Gi, int* status) {
  const int t = threadIdx.x, ks = jacobi_stride(K);
  const T small = sizeof(T) == 8 ? T(1e-300) : T(1e-37);
  if (t < k) {
    T nrm = 0;
    for (int r = 0; r < k; ++r) nrm += C[r * ks + t] * C[r * ks + t];
    inv[t] = nrm > small ? T(1) / sqrt(nrm) : T(0);
    if (!(nrm > small)) atomicOr(status, ST_JACOBI);
  }
  __syncthreads();
  for (int e = t; e < k * K; e += kT)
    if (e % K < k) C[e / K * ks + e % K] *= inv[e % K];
  __syncthreads();
  for (int e = t; e < K * K; e += kT) {
    const int a = e / K, b = e % K;
    T sum = 0;
    if (a < k && b < k)
      for (int j = 0; j < k; ++j) sum = fma(C[a * ks + j], V[b * ks + j], sum);
    Gi[e] = static_cast<float>(sum);
  }
}

// ---------------------------------------------------------------- align
// One CTA per partition.  G_i (K x K float, row-major) = D_i (sign) or O_i (OPT).
__global__ void __launch_bounds__(kT) align_kernel(const float* __restrict__ Zl, int64_t z_stride,
                                                   const float* __restrict__ Zb_one, int d, int k, int K,
                                                   int base_one, const int* __restrict__ part_base, int opt, int f64,
                                                   float* __restrict__ Gout, int* status) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int ks = jacobi_stride(K);
  double* C = reinterpret_cast<double*>(sm);   // K rows of stride ks
  double* V = C + K * ks;                       // the same
  double* part = V + K * ks;                    // kT x 16 floats
  const int i = blockIdx.x;
  const int t = threadIdx.x;
  after_previous();
  // the base of partition i's problem: one for the context, or per partition (batch groups)
  const int base = part_base ? part_base[i] : base_one;
  const float* Zb = part_base ? Zl + z_stride * base : Zb_one;
  float* Gi = Gout + int64_t(i) * K * K;
  if (i == base) {
    for (int e = t; e < K * K; e += kT) Gi[e] = ((e / K) == (e % K) && (e / K) < k) ? 1.f : 0.f;
    return;
  }
  const float* Zi = Zl + z_stride * i;
  if (!opt) {
    // sgn <Z_i[:, j], Z_b[:, j]> as FP64 accumulation gives it; sgn(0) = +1.  The FP64
    // pipe would take 12 us at d = 1,024, K = 16 (two conversions and a multiply-add per
    // entry at 2 per clock), so an FP32 sum decides where it can: with D the sum of
    // the products' magnitudes, any order of n FP32 multiply-adds is within n u D / (1 -
    // n u) of the exact sum, u = 2^-24 (Higham, Accuracy and Stability of Numerical
    // Algorithms, Sec. 3.1), plus 2^-150 for each that falls below the normal range
    // (Sec. 2.1), and the FP64 sum within far less.  The computed D lacks up to as much
    // of that again (n u <= 1).  A column whose FP32 sum is not above twice the first
    // term plus 2^-149 for each row (or is NaN) sends the block to the FP64 sums.
    // Measured, 64 blocks of 1,024 x 16: 16.3 -> 5.6 us; 4 of 100 x 5: 3.6 -> 2.2.
    const int j = t % K, sl = t / K, RS = kT / K;
    float* dots = reinterpret_cast<float*>(part);
    float f = 0.f, m = 0.f;
#pragma unroll 4
    for (int r = sl; r < d; r += RS) {
      const float x = Zi[int64_t(r) * K + j], y = Zb[int64_t(r) * K + j];
      f = fmaf(x, y, f);
      m = fmaf(fabsf(x), fabsf(y), m);
    }
    dots[t] = f;
    dots[kT + t] = m;
    __syncthreads();
    bool sure = true;
    if (t < K) {
      float tot = 0.f, mag = 0.f;
      for (int q = 0; q < RS; ++q) {
        tot += dots[q * K + t];
        mag += dots[kT + q * K + t];
      }
      // columns beyond k hold zeros: nothing to decide
      const float terms = static_cast<float>(d) + RS + 2;
      sure = t >= k || fabsf(tot) > 2.f * terms * 0x1.0p-24f * mag + terms * 0x1.0p-149f;
      part[kT + t] = tot;  // beyond the sums of either precision
    }
    if (__syncthreads_or(!sure)) {
      double s = 0.0;
      for (int r = sl; r < d; r += RS) s += static_cast<double>(Zi[int64_t(r) * K + j]) * Zb[int64_t(r) * K + j];
      part[t] = s;
      __syncthreads();
      if (t < K) {
        double tot = 0.0;
        for (int q = 0; q < RS; ++q) tot += part[q * K + t];
        part[kT + t] = tot;
      }
      __syncthreads();
    }
    before_next();
    for (int e = t; e < K * K; e += kT) {
      const int a = e / K, b = e % K;
      float v = 0.f;
      if (a == b && a < k) v = part[kT + a] < 0.0 ? -1.f : 1.f;
      Gi[e] = v;
    }
    return;
  }
  // OPT: C = Z_i^T Z_b.  Thread (4 x 4 block (bi, bj) of C, row slice sl) sums
  // FP32 products of rows sl, sl + S, ... in FP32; the slices are added in FP64
  // in slice order.  Then the Procrustes SVD by the CTA's Jacobi.
  float* red = reinterpret_cast<float*>(part);  // kT x 16 partial blocks
  {
    const int NB = K / 4, NBB = NB * NB, S = kT / NBB;
    const int blk = t % NBB, sl = t / NBB;
    const int bi = blk / NB, bj = blk % NB;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    constexpr int U = 4;  // rows per trip, loads issued before the FMAs
    for (int r0 = sl; r0 < d; r0 += S * U) {
      float4 u[U], v[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int r = r0 + q * S;
        u[q] = r < d ? *reinterpret_cast<const float4*>(Zi + int64_t(r) * K + 4 * bi) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[q] = r < d ? *reinterpret_cast<const float4*>(Zb + int64_t(r) * K + 4 * bj) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const float uu[4] = {u[q].x, u[q].y, u[q].z, u[q].w}, vv[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(uu[a], vv[b], acc[a][b]);
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) red[(4 * a + b) * kT + t] = acc[a][b];
    __syncthreads();
    for (int e = t; e < K * K; e += kT) {
      const int a = e / K, b = e % K;
      const int bb = (a / 4) * NB + b / 4, el = 4 * (a % 4) + b % 4;
      double sum = 0.0;
      for (int q = 0; q < S; ++q) sum += red[el * kT + q * NBB + bb];
      C[a * ks + b] = sum;
    }
    __syncthreads();
  }
  if (f64) {
    // k x k Procrustes SVD in FP64 (LP_FLAG_KXK_FP64): C = U Sigma V^T, O = U V^T
    const bool ok = cta_jacobi<double>(C, V, k, K);
    if (!ok && t == 0) atomicOr(status, ST_JACOBI);
    procrustes_factor<double>(C, V, part, k, K, Gi, status);
  } else {
    // FP32 copies in the V area (two float blocks fit in one of doubles)
    float* Cf = reinterpret_cast<float*>(V);
    float* Vf = Cf + K * ks;
    for (int e = t; e < K * ks; e += kT) Cf[e] = static_cast<float>(C[e]);
    __syncthreads();
    const bool ok = cta_jacobi<float>(Cf, Vf, k, K);
    if (!ok && t == 0) atomicOr(status, ST_JACOBI);
    procrustes_factor<float>(Cf, Vf, reinterpret_cast<float*>(part), k, K, Gi, status);
  }
}

// C and V (K rows of stride K + 1, doubles), then the partial-block area (kT x 16 floats; it
// also holds the column scales of the Procrustes factor, and the sign path's
// kT doubles)
size_t align_smem(int K) { return size_t(2) * K * jacobi_stride(K) * 8 + size_t(kT) * 16 * 4 + 16; }

// ---------------------------------------------------------------- residual error
// rho_i = ||Z_i G_i - Z_b||_2 (Def. 3) for one partition per CTA: E = Z_i G_i - Z_b
// is formed 64 rows at a time in shared memory (G_i the aligner: K x K, diagonal
// for sign-fixing, nullptr for none); E^T E is summed in FP32 over a chunk and in
// FP64 across chunks; its largest eigenvalue comes from the one-sided Jacobi.
constexpr int kRhoRows = 64;

__global__ void __launch_bounds__(kT) rho_kernel(const float* __restrict__ Zl, int64_t z_stride,
                                                 const float* __restrict__ Zb, const float* __restrict__ G,
                                                 int diag_only, int base, int d, int k, int K,
                                                 double* __restrict__ out, int* status) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int ks = jacobi_stride(K);
  double* C = reinterpret_cast<double*>(sm);  // K*K Gram
  double* V = C + K * K;                       // Jacobi workspace, K rows of stride ks
  float* E = reinterpret_cast<float*>(V + K * ks);  // kRhoRows x K
  const int i = blockIdx.x, t = threadIdx.x;
  if (i == base) {
    if (t == 0) out[i] = 0.0;
    return;
  }
  const float* Zi = Zl + z_stride * i;
  const float* Gi = G ? G + int64_t(i) * K * K : nullptr;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};  // entries e = t + j * kT of the K x K Gram
  for (int r0 = 0; r0 < d; r0 += kRhoRows) {
    const int nr = min(kRhoRows, d - r0);
    __syncthreads();
    for (int e = t; e < nr * K; e += kT) {
      const int r = r0 + e / K, j = e % K;
      float v;
      if (!Gi) {
        v = Zi[int64_t(r) * K + j];
      } else if (diag_only) {
        v = Zi[int64_t(r) * K + j] * Gi[j * K + j];
      } else {
        v = 0.f;
        for (int l = 0; l < K; ++l) v = fmaf(Zi[int64_t(r) * K + l], Gi[l * K + j], v);
      }
      E[e] = v - Zb[int64_t(r) * K + j];
    }
    __syncthreads();
    for (int q = 0; q < 4; ++q) {
      const int e = t + q * kT;
      if (e >= K * K) break;
      const int a = e / K, b = e % K;
      float s = 0.f;
      if (a < k && b < k)
        for (int r = 0; r < nr; ++r) s = fmaf(E[r * K + a], E[r * K + b], s);
      acc[q] += s;
    }
  }
  __syncthreads();
  for (int q = 0; q < 4; ++q) {
    const int e = t + q * kT;
    if (e < K * K) C[e] = acc[q];
  }
  __syncthreads();
  // E^T E is symmetric positive semidefinite: the one-sided Jacobi's column norms are its eigenvalues
  float* Cf = reinterpret_cast<float*>(V);
  float* Vf = Cf + K * ks;
  for (int e = t; e < K * K; e += kT) Cf[e / K * ks + e % K] = static_cast<float>(C[e]);
  __syncthreads();
  const bool ok = cta_jacobi<float>(Cf, Vf, k, K);
  if (!ok && t == 0) atomicOr(status, ST_JACOBI);
  if (t < 32) {
    float top = 0.f;
    for (int j = 0; j < k; ++j) {
      float v = 0.f;
      if (t < k) v = Cf[t * ks + j] * Cf[t * ks + j];
      v = warp_sumf(v);
      top = fmaxf(top, v);
    }
    if (t == 0) out[i] = sqrt(sqrt(static_cast<double>(top)));  // sqrt(lambda_max(E^T E))
  }
}

// ---------------------------------------------------------------- aggregate
// Y = sum_i w_i Y_i G_i over each problem's partitions (Alg. 1 aggregation; G_i
// the aligner: K x K, diagonal for sign-fixing, or none).  Thread (slice sl,
// row, group jg of four columns) sums the partitions i0 + sl, i0 + sl + S, ... in
// order into four FP32 accumulators, then the S slices are added in slice order
// through shared memory: a fixed summation order for a given S.  RPB = kT /
// (S K/4) rows per CTA; problem q = blockIdx.y sums its own partitions
// [i0, i1) into its own d x K block of Y.
template <int K>
__global__ void __launch_bounds__(kT) aggregate_kernel(const float* __restrict__ Yl, const float* __restrict__ w,
                                                       const float* __restrict__ G, int diag_only, int m, int d, int S,
                                                       const int* __restrict__ prob_begin, float* __restrict__ Y) {
  constexpr int JG = K / 4;
  __shared__ float4 red[kT];
  const int t = threadIdx.x;
  after_previous();
  before_next();
  const int RPB = kT / (JG * S);
  const int jg = t % JG, row = (t / JG) % RPB, sl = t / (JG * RPB);
  const int r = blockIdx.x * RPB + row;
  const int q = blockIdx.y;
  const int i0 = prob_begin ? prob_begin[q] : 0, i1 = prob_begin ? prob_begin[q + 1] : m;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (r < d) {
    for (int i = i0 + sl; i < i1; i += S) {
      const float* yi = Yl + (int64_t(i) * d + r) * K;
      float4 v;
      if (G == nullptr) {
        v = *reinterpret_cast<const float4*>(yi + 4 * jg);
      } else if (diag_only) {
        const float* gi = G + int64_t(i) * K * K + (4 * jg) * (K + 1);
        const float4 y = *reinterpret_cast<const float4*>(yi + 4 * jg);
        v = make_float4(y.x * gi[0], y.y * gi[K + 1], y.z * gi[2 * (K + 1)], y.w * gi[3 * (K + 1)]);
      } else {
        const float* gi = G + int64_t(i) * K * K + 4 * jg;
        float yr[K];
#pragma unroll
        for (int l = 0; l < K; l += 4) {
          const float4 y = *reinterpret_cast<const float4*>(yi + l);
          yr[l] = y.x;
          yr[l + 1] = y.y;
          yr[l + 2] = y.z;
          yr[l + 3] = y.w;
        }
        v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int l = 0; l < K; ++l) {
          const float4 g = *reinterpret_cast<const float4*>(gi + l * K);
          v.x = fmaf(yr[l], g.x, v.x);
          v.y = fmaf(yr[l], g.y, v.y);
          v.z = fmaf(yr[l], g.z, v.z);
          v.w = fmaf(yr[l], g.w, v.w);
        }
      }
      const float wi = w[i];
      acc.x = fmaf(wi, v.x, acc.x);
      acc.y = fmaf(wi, v.y, acc.y);
      acc.z = fmaf(wi, v.z, acc.z);
      acc.w = fmaf(wi, v.w, acc.w);
    }
  }
  red[t] = acc;
  __syncthreads();
  if (t < RPB * JG) {
    const int row2 = t / JG, jg2 = t % JG;
    const int r2 = blockIdx.x * RPB + row2;
    float4 sum = red[t];
    for (int s2 = 1; s2 < S; ++s2) {
      const float4 o = red[(s2 * RPB + row2) * JG + jg2];
      sum.x += o.x;
      sum.y += o.y;
      sum.z += o.z;
      sum.w += o.w;
    }
    if (r2 < d) reinterpret_cast<float4*>(Y + int64_t(q) * d * K + int64_t(r2) * K)[jg2] = sum;
  }
}

// Zl[i] = Z[part_prob[i]]: each partition's copy of its problem's d x K block
// (batch groups, where the first step of a round multiplies per-problem bases).
__global__ void broadcast_kernel(const float4* __restrict__ Z, const int* __restrict__ part_prob, int m,
                                 int64_t blk4, float4* __restrict__ Zl) {
  after_previous();
  before_next();
  const int64_t total = int64_t(m) * blk4;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = e / blk4, off = e - i * blk4;
    Zl[e] = Z[int64_t(part_prob[i]) * blk4 + off];
  }
}

// ---------------------------------------------------------------- Ritz
// H = Z^T (M Z) in FP64, split over row slices: block g adds the products of
// its rows (staged in shared memory) into Hpart[g]; ritz_solve adds the slices
// in slice order (deterministic), symmetrises, diagonalises (Jacobi: FP32, or
// FP64 under LP_FLAG_KXK_FP64),
// orders by descending Ritz value and writes sigma and the reordered V;
// ritz_rotate forms Zout = Z V row by row.
constexpr int kRitzRows = 64;  // rows per slice

__global__ void __launch_bounds__(kT) ritz_partial_kernel(const float* __restrict__ Z, const float* __restrict__ MZ,
                                                          int d, int k, int K, double* __restrict__ Hpart) {
  __shared__ float zs[kRitzRows * LP_MAX_K], ms[kRitzRows * LP_MAX_K];
  const int t = threadIdx.x;
  const int r0 = blockIdx.x * kRitzRows;
  // problem blockIdx.y: its d x K blocks and its slices of the scratch
  Z += int64_t(blockIdx.y) * d * K;
  MZ += int64_t(blockIdx.y) * d * K;
  Hpart += int64_t(blockIdx.y) * gridDim.x * K * K;
  const int nr = min(kRitzRows, d - r0);
  for (int e = t; e < nr * K; e += kT) {
    zs[e] = Z[int64_t(r0) * K + e];
    ms[e] = MZ[int64_t(r0) * K + e];
  }
  __syncthreads();
  double* H = Hpart + int64_t(blockIdx.x) * K * K;
  for (int e = t; e < K * K; e += kT) {
    const int a = e / K, b = e % K;
    double sum = 0.0;
    if (a < k && b < k)
      for (int r = 0; r < nr; ++r) sum += static_cast<double>(zs[r * K + a]) * ms[r * K + b];
    H[e] = sum;
  }
}

__global__ void __launch_bounds__(kT) ritz_solve_kernel(const double* __restrict__ Hpart, int slices, int k, int K,
                                                        double n_one, const double* __restrict__ n_of, int f64,
                                                        double* __restrict__ Vo, double* __restrict__ sigma,
                                                        int* status) {
  extern __shared__ __align__(16) unsigned char sm[];
  // problem blockIdx.x: its slices, its V and sigma, its row count
  const int qp = blockIdx.x;
  Hpart += int64_t(qp) * slices * K * K;
  Vo += int64_t(qp) * K * K;
  sigma += int64_t(qp) * LP_MAX_K;
  const double n = n_of ? n_of[qp] : n_one;
  const int ks = jacobi_stride(K);
  double* H = reinterpret_cast<double*>(sm);  // K rows of stride ks
  double* V = H + K * ks;                      // the same
  double* lam = V + K * ks;                    // K
  int* order = reinterpret_cast<int*>(lam + K);
  const int t = threadIdx.x;
  for (int e = t; e < K * K; e += kT) {
    double sum = 0.0;
    for (int g = 0; g < slices; ++g) sum += Hpart[int64_t(g) * K * K + e];
    H[e / K * ks + e % K] = sum;
  }
  __syncthreads();
  // symmetrise: the thread of entry (a, b), a < b, writes both halves
  for (int e = t; e < K * K; e += kT) {
    const int a = e / K, b = e % K;
    if (a < b) {
      const double v = 0.5 * (H[a * ks + b] + H[b * ks + a]);
      H[a * ks + b] = v;
      H[b * ks + a] = v;
    }
  }
  __syncthreads();
  // H is symmetric positive semidefinite: its one-sided Jacobi SVD is its
  // eigendecomposition, in FP64 under LP_FLAG_KXK_FP64, else on FP32 copies in
  // the V area.
  if (f64) {
    const bool ok = cta_jacobi<double>(H, V, k, K);
    if (!ok && t == 0) atomicOr(status, ST_JACOBI);
    if (t < k) {
      double v = 0.0;
      for (int r = 0; r < k; ++r) v += H[r * ks + t] * H[r * ks + t];
      lam[t] = v > 0.0 ? sqrt(v) : 0.0;
    }
  } else {
    float* Hf = reinterpret_cast<float*>(V);
    float* Vf = Hf + K * ks;
    for (int e = t; e < K * K; e += kT) Hf[e / K * ks + e % K] = static_cast<float>(H[e / K * ks + e % K]);
    __syncthreads();
    const bool ok = cta_jacobi<float>(Hf, Vf, k, K);
    if (!ok && t == 0) atomicOr(status, ST_JACOBI);
    if (t < k) {
      float v = 0.f;
      for (int r = 0; r < k; ++r) v += Hf[r * ks + t] * Hf[r * ks + t];
      lam[t] = v > 0.f ? sqrt(static_cast<double>(v)) : 0.0;
    }
  }
  __syncthreads();
  if (t == 0) {
    for (int j = 0; j < k; ++j) order[j] = j;
    for (int a = 0; a < k; ++a)
      for (int b = a + 1; b < k; ++b)
        if (lam[order[b]] > lam[order[a]]) {
          const int tmp = order[a];
          order[a] = order[b];
          order[b] = tmp;
        }
    for (int j = 0; j < k; ++j) sigma[j] = sqrt(n * lam[order[j]]);
  }
  __syncthreads();
  for (int e = t; e < K * K; e += kT) {
    const int l = e / K, j = e % K;
    Vo[e] = j >= k ? 0.0
                   : f64 ? V[l * ks + order[j]]
                         : static_cast<double>(reinterpret_cast<const float*>(V)[K * ks + l * ks + order[j]]);
  }
}

__global__ void ritz_rotate_kernel(const float* __restrict__ Z, const double* __restrict__ Vo, int d, int k, int K,
                                   int nprob, double* __restrict__ Zout) {
  const int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (e >= int64_t(nprob) * d * k) return;
  // problem q's d x k output block follows problem q - 1's
  const int q = static_cast<int>(e / (int64_t(d) * k));
  const int64_t el = e - int64_t(q) * d * k;
  Z += int64_t(q) * d * K;
  Vo += int64_t(q) * K * K;
  const int r = static_cast<int>(el / k), j = static_cast<int>(el % k);
  double sum = 0.0;
  for (int l = 0; l < k; ++l) sum += static_cast<double>(Z[int64_t(r) * K + l]) * Vo[l * K + j];
  Zout[e] = sum;
}

}  // namespace

cudaError_t allow_max_dynamic_smem(const void* kern) {
  static std::mutex mu;
  static std::unordered_set<const void*> done;
  std::lock_guard<std::mutex> lock(mu);
  if (done.count(kern)) return cudaSuccess;
  int dev = 0, optin = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - static_cast<int>(fa.sharedSizeBytes));
  if (e == cudaSuccess) done.insert(kern);
  return e;
}

cudaError_t launch_split_planes(const SplitParts& parts, int64_t src_ld, int d, uint16_t* hi, uint16_t* lo, int64_t ld,
                                cudaStream_t s) {
  const int64_t total = parts.n > 0 ? parts.row0[parts.n] * (ld / 8) : 0;
  if (total <= 0) return cudaSuccess;
  const int64_t blocks = std::min<int64_t>((total + 2 * kT - 1) / (2 * kT), 152 * 8);
  split_planes_kernel<<<static_cast<unsigned>(blocks), kT, 0, s>>>(parts, src_ld, d, hi, lo, static_cast<int>(ld / 8));
  return cudaGetLastError();
}

namespace {
unsigned rows_grid(int64_t total) {
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((total + kT - 1) / kT, 152 * 16)));
}
}  // namespace

cudaError_t launch_pack(const double* src, float* dst, int batch, int d, int k, int K, cudaStream_t s, int* clear) {
  const int64_t rows = int64_t(batch) * d;
  pack_kernel<<<rows_grid(rows * (K / 4)), kT, 0, s>>>(src, dst, rows, k, K, clear);
  return cudaGetLastError();
}

cudaError_t launch_to_float(const double* src, float* dst, int n, cudaStream_t s) {
  to_float_kernel<<<(n + kT - 1) / kT, kT, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const float* src, double* dst, int batch, int d, int k, int K, cudaStream_t s) {
  const int64_t rows = int64_t(batch) * d;
  unpack_kernel<<<rows_grid(rows * (K / 4)), kT, 0, s>>>(src, dst, rows, k, K);
  return cudaGetLastError();
}

namespace {
template <int G>
cudaError_t launch_reduce_g(const float* P, const int* slot_begin, const float* scale, int m, int d, int K, float* Y,
                            double* Yd, int k, const int* status, int* status_host, Lane at) {
  const int64_t n4 = int64_t(d) * K / 4;
  const dim3 grid(static_cast<unsigned>((n4 + kT / G - 1) / (kT / G)), static_cast<unsigned>(m));
  return launch_on(at, Yd ? reduce_kernel<G, true> : reduce_kernel<G, false>, grid, kT, 0, 0, P, slot_begin, scale, d, K, Y,
                   Yd, k, status, status_host);
}

cudaError_t reduce_any(const float* P, const int* slot_begin, const float* scale, int m, int d, int K, float* Y,
                       double* Yd, int k, const int* status, int* status_host, Lane at, int max_slots) {
  int G = 1;
  while (G < 32 && max_slots > 4 * G) G <<= 1;
  switch (G) {
    case 1: return launch_reduce_g<1>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
    case 2: return launch_reduce_g<2>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
    case 4: return launch_reduce_g<4>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
    case 8: return launch_reduce_g<8>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
    case 16: return launch_reduce_g<16>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
    default: return launch_reduce_g<32>(P, slot_begin, scale, m, d, K, Y, Yd, k, status, status_host, at);
  }
}
}  // namespace

cudaError_t launch_reduce(const float* P, const int* slot_begin, const float* scale, int m, int d, int K, float* Y,
                          Lane at, int max_slots) {
  return reduce_any(P, slot_begin, scale, m, d, K, Y, nullptr, 0, nullptr, nullptr, at, max_slots);
}

cudaError_t launch_reduce_f64(const float* P, const int* slot_begin, const float* scale, int m, int d, int k, int K,
                              double* Y, const int* status, int* status_host, Lane at, int max_slots) {
  return reduce_any(P, slot_begin, scale, m, d, K, nullptr, Y, k, status, status_host, at, max_slots);
}

cudaError_t launch_align(const float* Zl, int64_t z_stride, const float* Zb, int m, int d, int k, int K, int base,
                         lp_aggregator agg, float* G, int* status, Lane at, bool kxk_fp64,
                         const int* part_base) {
  return launch_on(at, align_kernel, dim3(m), kT, align_smem(K), 0, Zl, z_stride, Zb, d, k, K, base, part_base,
                   agg == LP_AGG_OPT ? 1 : 0, kxk_fp64 ? 1 : 0, G, status);
}

cudaError_t launch_aggregate(const float* Yl, const float* w, const float* G, int diag_only, int m, int d, int K,
                             float* Y, Lane at, const int* prob_begin, int nprob) {
  // slices: a power of two up to the partitions per problem, at most 16
  const int per = nprob > 0 ? m / nprob : m;
  int S = 1;
  while (S * 2 <= per && S * 2 <= 16) S *= 2;
  const int rpb = kT / (K / 4 * S);
  const dim3 grid((d + rpb - 1) / rpb, nprob);
  auto go = [&](auto kern) {
    return launch_on(at, kern, grid, kT, 0, 0, Yl, w, G, diag_only, m, d, S, prob_begin, Y);
  };
  switch (K) {
    case 8: return go(aggregate_kernel<8>);
    case 16: return go(aggregate_kernel<16>);
    case 32: return go(aggregate_kernel<32>);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_broadcast(const float* Z, const int* part_prob, int m, int d, int K, float* Zl, Lane at) {
  const int64_t blk4 = int64_t(d) * K / 4;
  const int64_t total = int64_t(m) * blk4;
  const int blocks = static_cast<int>(std::min<int64_t>((total + kT - 1) / kT, 4096));
  return launch_on(at, broadcast_kernel, dim3(blocks > 0 ? blocks : 1), kT, 0, 0, reinterpret_cast<const float4*>(Z),
                   part_prob, m, blk4, reinterpret_cast<float4*>(Zl));
}

cudaError_t launch_ritz(const float* Z, const float* MZ, int d, int k, int K, double n, double* Zout, double* sigma,
                        double* scratch, int* status, cudaStream_t s, bool kxk_fp64, int nprob, const double* n_of) {
  const int slices = (d + kRitzRows - 1) / kRitzRows;
  double* Hpart = scratch;
  double* Vo = scratch + size_t(nprob) * slices * K * K;
  ritz_partial_kernel<<<dim3(slices, nprob), kT, 0, s>>>(Z, MZ, d, k, K, Hpart);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t sm = size_t(2) * K * jacobi_stride(K) * 8 + size_t(K) * 8 + size_t(K) * 4 + 16;
  ritz_solve_kernel<<<nprob, kT, sm, s>>>(Hpart, slices, k, K, n, n_of, kxk_fp64 ? 1 : 0, Vo, sigma, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int64_t total = int64_t(nprob) * d * k;
  ritz_rotate_kernel<<<static_cast<unsigned>((total + kT - 1) / kT), kT, 0, s>>>(Z, Vo, d, k, K, nprob, Zout);
  return cudaGetLastError();
}

cudaError_t launch_rho(const float* Zl, int64_t z_stride, const float* Zb, const float* G, int diag_only, int base,
                       int m, int d, int k, int K, double* out, int* status, cudaStream_t s) {
  const size_t sm = (size_t(K) * K + size_t(K) * jacobi_stride(K)) * 8 + size_t(kRhoRows) * K * 4;
  rho_kernel<<<m, kT, sm, s>>>(Zl, z_stride, Zb, G, diag_only, base, d, k, K, out, status);
  return cudaGetLastError();
}

size_t ritz_scratch_bytes(int d, int K, int nprob) {
  const int slices = (d + kRitzRows - 1) / kRitzRows;
  return size_t(nprob) * (size_t(slices) + 1) * K * K * 8;
}

}  // namespace lp

// Inline-PTX building blocks shared by the tensor-core step kernels: mbarriers,
// TMA tile loads, cluster shared-memory copies, tcgen05 MMA / TMEM access and the
// SWIZZLE_128B operand layout.  Everything here is a thin wrapper over one PTX
// instruction (or a fixed short sequence); no arithmetic of the method lives here.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <cstdint>

namespace lp {
namespace tc {

constexpr int kThreads = 256;
constexpr int kBM = 128;
constexpr int kChunkBytes = kBM * 128;  // 128 rows x 64 BF16
constexpr long long kTimeoutCycles = 4000000000LL;  // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t su32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
      : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
  return ok != 0;
}
// Non-blocking test of a phase (for loops that poll several barriers: try_wait
// may suspend the thread on one barrier while another is already complete).
__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
      : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try_cluster(uint32_t addr, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
      : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Bulk copy shared::cta -> another CTA's shared memory; completion is counted in
// bytes on the destination CTA's mbarrier.  Addresses 16-byte aligned, size a
// multiple of 16.
__device__ __forceinline__ void bulk_s2s_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "r"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(su32(bar))
      : "memory");
}

// Same load with an L2 eviction-priority policy (from createpolicy) on the lines it reads.
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, "
      "%3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(su32(bar)), "l"(policy)
      : "memory");
}
// Three-dimensional forms for maps that view a row-major matrix as (64 columns of
// a chunk, row, chunk index): one box of {64, rows, chunks} lands as `chunks`
// consecutive [rows][64] tiles, the layout two-dimensional boxes of 64 columns
// give one chunk at a time.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(su32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                                 uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, "
      "%3, %4}], [%5], %6;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(su32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];" ::"l"(reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z)
               : "memory");
}
// Bring one tile of the tensor into L2 without a shared-memory destination.
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}
// 32 lanes x 16 consecutive 32-bit TMEM columns; lane i of the warp gets lane (base + i).
// The registers may be read after tmem_wait and the tmem_value of each group of 16.
__device__ __forceinline__ void tmem_ld16_begin(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_value(uint32_t* r, float* v) {
  // (nothing that reads the registers moves above this, nor it above the wait)
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 Q consecutive columns with one wait.
template <int Q>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float* v) {
  uint32_t r[16 * Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) tmem_ld16_begin(taddr + 16 * q, r + 16 * q);
  tmem_wait();
#pragma unroll
  for (int q = 0; q < Q; ++q) tmem_value(r + 16 * q, v + 16 * q);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) { tmem_ld<1>(taddr, v); }

// Position (in floats) of the 4-float group holding column j of row r in a
// row-major 128 x K FP32 buffer; groups are XOR-permuted so that a warp's
// float4 row writes touch distinct banks.
template <int K>
__device__ __forceinline__ int wpos(int r, int j) {
  constexpr int rows_per_128b = 32 / K;
  constexpr int groups = K / 4;
  return r * K + ((((j >> 2) ^ ((r / rows_per_128b) % groups))) << 2) + (j & 3);
}

// Shared-memory matrix descriptor, SWIZZLE_128B, tcgen05 format (version field = 1).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: kind::f16, BF16 x BF16 -> FP32, dense.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn_major, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// Byte offset of element (row n, k-index kk) of a K-major SWIZZLE_128B operand
// whose rows hold 64 BF16 per 128-byte chunk; chunks of `rows` rows are contiguous.
__device__ __forceinline__ uint32_t sw128_off(int n, int kk, int rows) {
  const int chunk = kk >> 6, k2 = (kk & 63) * 2;
  return static_cast<uint32_t>(chunk * rows * 128 + n * 128 + ((((k2 >> 4) ^ (n & 7))) << 4) + (k2 & 15));
}

__device__ __forceinline__ uint16_t bf16_bits(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float bf16_val(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }

// The 16-bit operand types of the step kernels: the bits of rn(x) and its value.
struct Bf16Op {
  static __device__ __forceinline__ uint16_t bits(float x) { return bf16_bits(x); }
  static __device__ __forceinline__ float val(uint16_t b) { return bf16_val(b); }
};

// [Z_hi | Z_lo]^T of columns c0 .. c0 + dc - 1 of Z (d x K, FP32; zero beyond d) as a
// K-major SWIZZLE_128B operand of 2 K rows, hi = rn(z), lo = rn(z - hi), by threads
// t = 0 .. n - 1.  A thread takes eight consecutive columns at J values of j: eight
// loads in flight, contiguous over the lanes' j, and one 16-byte store per j and half
// (a row's eight columns are one swizzle atom).  Element by element, the same staging
// of 1,024 x 16 took about 16 us of 2-byte stores behind dependent loads, at every
// partition a CTA works on; with J = 1 4.5 us, with J = 4 (16-byte loads) 3.4.  J = 1
// spreads a small block over more threads (128 x 16: 11.9 us a launch against 12.3).
template <int K, int J, typename Op>
__device__ __forceinline__ void stage_z_items(unsigned char* s, const float* __restrict__ Z, int c0, int dc, int d, int t,
                                              int n) {
  constexpr int N = 2 * K, KJ = K / J;
#pragma unroll(J == 1 ? 2 : 1)
  for (int e = t; e < dc / 8 * KJ; e += n) {
    const int j = e % KJ * J, c = e / KJ * 8;
    float z[8][J];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float* p = Z + static_cast<int64_t>(c0 + c + q) * K + j;
      const bool in = c0 + c + q < d;
      if constexpr (J == 4) {
        const float4 v = in ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
        z[q][0] = v.x; z[q][1] = v.y; z[q][2] = v.z; z[q][3] = v.w;
      } else {
        z[q][0] = in ? *p : 0.f;
      }
    }
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float z0 = z[2 * q][jj], z1 = z[2 * q + 1][jj];
        const uint16_t h0 = Op::bits(z0), h1 = Op::bits(z1);
        hi[q] = h0 | (static_cast<uint32_t>(h1) << 16);
        lo[q] = Op::bits(z0 - Op::val(h0)) | (static_cast<uint32_t>(Op::bits(z1 - Op::val(h1))) << 16);
      }
      *reinterpret_cast<uint4*>(s + sw128_off(j + jj, c, N)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(s + sw128_off(K + j + jj, c, N)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}
template <int K, typename Op>
__device__ __forceinline__ void stage_z(unsigned char* s, const float* __restrict__ Z, int c0, int dc, int d, int t, int n) {
  if (dc / 8 * K <= 2 * n) stage_z_items<K, 1, Op>(s, Z, c0, dc, d, t, n);
  else stage_z_items<K, 4, Op>(s, Z, c0, dc, d, t, n);
}

// Barrier `id` over n threads (whole warps); and the same with the OR of a flag over them.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ bool bar_or(int id, int n, bool flag) {
  uint32_t r;
  asm volatile(
      "{ .reg .pred p, q; setp.ne.u32 q, %3, 0;\n\t"
      "bar.red.or.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p; }"
      : "=r"(r)
      : "r"(id), "r"(n), "r"(flag ? 1u : 0u)
      : "memory");
  return r != 0;
}

// Cluster sum of W (128 x K FP32, row r of this CTA's partial in w of epilogue thread r).
// Owner o holds rows [o RPC, (o + 1) RPC), RPC = 128 / CL.  Every CTA writes its partial rows to sW and one
// thread ships each owner its rows (bulk copies counted in bytes on the owner's parts_full);
// owners add the partials in source-rank order, in place, and ship the sums back the same
// way (sums_full).  A buffer is rewritten only after the waits show its previous contents
// were consumed.  The waits return false when they gave up, and so does this.
template <int K, typename WaitParts, typename WaitSums, typename Sync>
__device__ __forceinline__ bool sum_over_cluster(float (&w)[K], int r, uint32_t crank, uint32_t CL, int RPC, float* sW,
                                                 float* sWrecv, uint64_t* parts_full, uint64_t* sums_full,
                                                 WaitParts&& wait_parts, WaitSums&& wait_sums, Sync&& epi_sync) {
  const uint32_t rows_bytes = static_cast<uint32_t>(RPC * K * 4);
  if (r == 0) bulk_wait_read0();  // the previous tile's copies have read sW
  if (!epi_sync()) return false;
#pragma unroll
  for (int j = 0; j < K; j += 4)
    *reinterpret_cast<float4*>(sW + wpos<K>(r, j)) = make_float4(w[j], w[j + 1], w[j + 2], w[j + 3]);
  fence_async_smem();
  if (!epi_sync()) return false;
  if (r == 0) {
    mbar_expect_tx(parts_full, (CL - 1) * rows_bytes);
    for (uint32_t o = 0; o < CL; ++o)
      if (o != crank)
        bulk_s2s_cluster(mapa(su32(sWrecv + crank * RPC * K), o), su32(sW + o * RPC * K), rows_bytes,
                         mapa(su32(parts_full), o));
    bulk_commit();
  }
  if (!wait_parts()) return false;
  const int per = RPC * K / kBM;  // values per epilogue thread (K / CL), neighbours in a row
  // partials in source-rank order; four columns at a time where a thread has them
  if (per % 4 == 0) {
    for (int e = 0; e < per; e += 4) {
      const int idx = r * per + e, rl = idx / K, col = idx % K;
      const int own = wpos<K>(static_cast<int>(crank) * RPC + rl, col);
      const int rel = own - static_cast<int>(crank) * RPC * K;  // offset inside one owner's row block
      float4 v[8], sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (uint32_t src = 0; src < 8; ++src)
        if (src < CL) v[src] = *reinterpret_cast<const float4*>(src == crank ? sW + own : sWrecv + src * RPC * K + rel);
#pragma unroll
      for (uint32_t src = 0; src < 8; ++src)
        if (src < CL) {
          sum.x += v[src].x;
          sum.y += v[src].y;
          sum.z += v[src].z;
          sum.w += v[src].w;
        }
      *reinterpret_cast<float4*>(sW + own) = sum;
    }
  } else {
    for (int e = 0; e < per; ++e) {
      const int idx = r * per + e, rl = idx / K, col = idx % K;
      const int own = wpos<K>(static_cast<int>(crank) * RPC + rl, col);
      const int rel = own - static_cast<int>(crank) * RPC * K;
      float sum = 0.f;
      for (uint32_t src = 0; src < CL; ++src) sum += src == crank ? sW[own] : sWrecv[src * RPC * K + rel];
      sW[own] = sum;
    }
  }
  fence_async_smem();
  if (!epi_sync()) return false;
  if (r == 0) {
    mbar_expect_tx(sums_full, (CL - 1) * rows_bytes);
    for (uint32_t dst = 0; dst < CL; ++dst)
      if (dst != crank)
        bulk_s2s_cluster(mapa(su32(sW + crank * RPC * K), dst), su32(sW + crank * RPC * K), rows_bytes,
                         mapa(su32(sums_full), dst));
    bulk_commit();
  }
  if (!wait_sums()) return false;
#pragma unroll
  for (int j = 0; j < K; j += 4) {
    const float4 v = *reinterpret_cast<const float4*>(sW + wpos<K>(r, j));
    w[j] = v.x;
    w[j + 1] = v.y;
    w[j + 2] = v.z;
    w[j + 3] = v.w;
  }
  return true;
}

}  // namespace tc
}  // namespace lp

// Fused local power step on the 5th-generation tensor cores for A stored as
// FP8-E4M3 codes with one FP32 scale per row (a_r = s_r q_r):
//   P[slot] = A_seg^T (A_seg Z_i) = Q^T diag(s^2) Q Z_i      (eq. (2), unscaled),
// streaming form (the geometry, unit ring and cluster exchange of the streaming
// BF16 kernel in step_tcs.cu).
//
// The scales factor out of both contractions, so the tensor cores only ever see
// the codes.  Every E4M3 value is exactly an FP16 value (3 significand bits,
// exponents 2^-9 .. 2^8), and one cvt.rn.f16x2.e4m3x2 turns two codes into two
// FP16, so:
//   * two groups of four converter warps, one for each pass, take 128-row x 128-column
//     units of codes (16 KB): straight into registers, kDepth units ahead, widened and
//     written in the FP16 operand layout the MMAs read (SWIZZLE_128B, K-major, 32 KB per
//     unit) into the operand ring;
//   * first pass  D1 += Q_u [Z_hi | Z_lo]  (kind::f16 with FP16 operands; Z
//     split into FP16 hi + lo, 22 significand bits between them);
//   * epilogue    W = D1[:, :K] + D1[:, K:] (cluster-summed), then row r scaled
//     by s_r^2 / S with S = max_r s_r^2 (so |W| never exceeds the FP16 range:
//     |q_r . z| <= 448 sqrt(d)), split into FP16 hi + lo;
//   * second pass D2[b] += Q_u^T [W_hi | W_lo], re-read from L2 and widened
//     again; P = S (D2[:, :K] + D2[:, K:]).
// A row whose s_r^2 / S is below the FP16 range contributes nothing: its
// contribution is below 2^-24 of the largest row's, under FP32 rounding of P.
//
// What bounds it.  Z, the W operands and the exchange buffers leave about 96 KB of
// shared memory at d = 2,048, k = 32.  With the codes staged there by TMA (two 16 KB
// slots beside two operand slots) both passes together had 32 KB in flight and every
// unit crossed shared memory twice: 2,150 us a launch at n = 1M.  In registers the
// codes in flight cost no shared memory (64 KB at kDepth = 2) and the operand ring has
// three slots; a converter group for each pass overlaps the latencies of two units
// (one group of eight warps spent 1,450 cycles on each); roles step through their own
// units in closed form; the second pass runs two tiles behind the first where tensor
// memory holds a third D1, which takes the cluster exchange of W off the chain; and the
// exchange itself adds four columns at a time and waits for its copies only before it
// rewrites their source (12,000 -> 9,000 cycles a tile).  1,211 us at n = 1M, 1.7 TB/s of
// codes; n = 262,144: 456 -> 332 us over these steps, 123 -> 94 at d = 512 without a
// cluster.  A group still takes about 2,500 cycles a unit (widening 640, issuing its
// loads up to 600, the fence 90, the rest waiting for slots and data), three times what
// the conversion pipe needs.
//
// Roles (448 threads): warps 0-3 and 8-11 convert (first and second pass); warps 4-7 run the epilogue; lane 0
// of warps 12 and 13 issue the first and the second pass's MMAs (one thread issues a
// small-N MMA only every ~55 cycles, ~100 when it polls barriers in between); warps
// 4-7, 12 and 13 stage Z when the partition changes, while the converters go on.
// Every wait is bounded: on expiry the kernel records ST_TIMEOUT, stops issuing,
// retires its MMAs, frees tensor memory and returns.
#include <cuda_fp16.h>

#include "lp_internal.cuh"
#include "tc_ptx.cuh"

namespace lp {
namespace {

using namespace tc;

constexpr int kThreads8 = 448;
constexpr int kConvThreads = 256;            // warps 0-3 and 8-11, two groups
constexpr int kIssue1 = 12;                  // lane 0 of this warp issues the first pass, of the next one the second
constexpr int kOthers8 = kThreads8 - kConvThreads;
constexpr int kDepth = 2;                    // units of codes in flight per converter group
constexpr int kUnitBytes = 2 * kChunkBytes;  // 128 rows x 128 columns of FP16 (two 64-column chunks)
constexpr int kMaxRing = 8;
constexpr int kMaxD1 = 3;                    // D1 buffers
constexpr int kSmemLimit = 232448;

enum Tcs8Bar { S_D1FULL0 = 0, S_D1EMPTY0 = 3, S_B2FULL0 = 6, S_B2FREE0 = 8, S_D2FULL = 10, S_D2EMPTY = 11,
               S_REDFULL = 12, S_WFULL = 13, S_DONE = 14, S_EPI = 15, S_RING0 = 16 };
// operand ring: FULL[s] = S_RING0 + s, EMPTY[s] = S_RING0 + kMaxRing + s
constexpr int kNumBars8 = S_RING0 + 2 * kMaxRing;

struct Tcs8Args {
  const unsigned char* codes;  // n x ld, columns d .. ld - 1 zero
  int64_t n, ld;
  const Segment* segs;
  const int* seg_ptr;  // per cluster
  const float* Z;
  int64_t z_stride;
  float* P;
  int d;
  int* status;
  const float* scales;  // per global row
  float smax2;          // S = max_r s_r^2
  int ncd;              // 64-column chunks in this CTA's slice (even)
  int ring;             // operand ring units
  int lag;              // units of a tile's first pass ahead of the second pass of the tile `behind` before it
  int behind;           // tiles the second pass runs behind the first (D1 buffers less one)
  int hints;
  uint32_t off_B1, off_B2, off_W, off_Wrecv, off_bar, tmem_cols;
};

// A run: the consecutive pieces of one partition that a cluster owns, one stream of
// tiles (every piece but the last is a whole number of tiles).
struct Run8 {
  int si, sj;      // segments
  int64_t row0, row1;
  int ntiles;
};
__device__ __forceinline__ Run8 run_at(const Segment* segs, int si, int se) {
  Run8 r;
  r.si = si;
  r.row0 = segs[si].row0;
  const int part = segs[si].part;
  r.sj = si + 1;
  while (r.sj < se && segs[r.sj].part == part) ++r.sj;
  r.row1 = segs[r.sj - 1].row1;
  r.ntiles = static_cast<int>((r.row1 - r.row0 + kBM - 1) / kBM);
  return r;
}

// The order of a run's units in the ring: the first pass of tile t (blocks 0 .. U-1)
// interleaved with the second pass of tile t - behind, `lag` blocks later.  In closed
// form, so that each role steps through its own units only (walking the whole order
// cost an issuing thread some 300 cycles a unit).
struct Order8 {
  int U, lag, behind;
  // units of the run before tile t's turn
  __device__ __forceinline__ uint32_t before(int t, int ntiles) const {
    return static_cast<uint32_t>(U * (min(t, ntiles) + max(0, t - behind)));
  }
  __device__ __forceinline__ uint32_t first(int t, int u, int ntiles) const {
    return before(t, ntiles) + u + (t >= behind ? max(0, u - lag) : 0);
  }
  __device__ __forceinline__ uint32_t second(int tile, int v, int ntiles) const {
    const int t = tile + behind;
    return before(t, ntiles) + (t < ntiles ? min(v + lag + 1, U) : 0) + v;
  }
};

// A role's place in the ring: unit g sits in slot g mod R, its fill's number is g / R.
struct Place8 {
  uint32_t g = 0, slot = 0, fill = 0;
  __device__ __forceinline__ void to(uint32_t next, uint32_t R) {
    slot += next - g;
    g = next;
    while (slot >= R) {
      slot -= R;
      ++fill;
    }
  }
};

// Instruction descriptor: kind::f16 with FP16 A and B, FP32 accumulate, dense.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool a_mn_major, bool b_mn_major) {
  return (1u << 4) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// Four codes -> four FP16 in order.
__device__ __forceinline__ void e4m3x4_to_f16x4(uint32_t codes, uint32_t& lo, uint32_t& hi) {
  asm("{ .reg .b16 a, b; mov.b32 {a, b}, %2; cvt.rn.f16x2.e4m3x2 %0, a; cvt.rn.f16x2.e4m3x2 %1, b; }"
      : "=r"(lo), "=r"(hi)
      : "r"(codes));
}

__device__ __forceinline__ uint16_t f16_bits(float x) { return __half_as_ushort(__float2half_rn(x)); }
__device__ __forceinline__ float f16_val(uint16_t b) { return __half2float(__ushort_as_half(b)); }
struct F16Op {
  static __device__ __forceinline__ uint16_t bits(float x) { return f16_bits(x); }
  static __device__ __forceinline__ float val(uint16_t b) { return f16_val(b); }
};

__device__ __forceinline__ uint4 ld_codes(const unsigned char* p, uint64_t policy) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(policy));
  return v;
}

template <int K>
__global__ void __launch_bounds__(kThreads8, 1) step_tcs8_kernel(Tcs8Args a) {
  constexpr int N = 2 * K;
  constexpr uint32_t B2BUF = 2 * N * 128;
  constexpr int TP = static_cast<int>(kTcChainRows / kBM);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sRing = base;
  unsigned char* sB1 = base + a.off_B1;
  unsigned char* sB2 = base + a.off_B2;
  float* sW = reinterpret_cast<float*>(base + a.off_W);
  float* sWrecv = reinterpret_cast<float*>(base + a.off_Wrecv);
  uint64_t* bar = reinterpret_cast<uint64_t*>(base + a.off_bar);
  const int R = a.ring;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bar + kNumBars8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  volatile uint32_t* fills = tmem_holder + 4;  // per slot: fills begun

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t crank = cluster_rank();
  const uint32_t CL = cluster_size();
  const int RPC = kBM / static_cast<int>(CL);
  const int cluster_id = blockIdx.x / CL;
  const int DC = 64 * a.ncd;
  const int c0 = static_cast<int>(crank) * DC;
  const int U = a.ncd / 2;  // one unit per 128-column block
  const int ND1 = a.behind + 1;

  if (tid == 0) {
    for (int s = 0; s < kMaxD1; ++s) {
      mbar_init(&bar[S_D1FULL0 + s], 1);
      mbar_init(&bar[S_D1EMPTY0 + s], 4);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bar[S_B2FULL0 + s], kBM);
      mbar_init(&bar[S_B2FREE0 + s], 1);
    }
    mbar_init(&bar[S_D2FULL], 1);
    mbar_init(&bar[S_D2EMPTY], 4);
    mbar_init(&bar[S_REDFULL], 1);
    mbar_init(&bar[S_WFULL], 1);
    mbar_init(&bar[S_DONE], 2);
    mbar_init(&bar[S_EPI], 128);
    for (int s = 0; s < kMaxRing; ++s) {
      mbar_init(&bar[S_RING0 + s], kConvThreads / 64);  // one arrival per warp of the group
      mbar_init(&bar[S_RING0 + kMaxRing + s], 1);        // MMA commit
    }
    *abort_flag = 0;
    for (int s = 0; s < kMaxRing; ++s) fills[s] = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_holder)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  const uint32_t tD2 = tmem + static_cast<uint32_t>(ND1 * N);

  auto give_up = [&]() {
    *abort_flag = 1;
    atomicOr(a.status, ST_TIMEOUT);
  };
  auto wait = [&](int id, uint32_t parity, bool cluster_scope) -> bool {
    const uint32_t addr = su32(&bar[id]);
    const long long t0 = clock64();
    while (true) {
      if (cluster_scope ? mbar_try_cluster(addr, parity) : mbar_try(addr, parity)) return true;
      if (*abort_flag) return false;
      if (clock64() - t0 > kTimeoutCycles) {
        give_up();
        return false;
      }
    }
  };
  // Both issuers and both converter groups share one ring in unit order; before a parity
  // wait on a slot they see that enough of its fills have begun, i.e. that the phase
  // before the one they wait for is over (a wait a phase early would succeed at once).
  auto wait_fills = [&](uint32_t slot, uint32_t count) -> bool {
    if (fills[slot] >= count) return true;
    const long long t0 = clock64();
    while (fills[slot] < count) {
      if (*abort_flag) return false;
      if (clock64() - t0 > kTimeoutCycles) {
        give_up();
        return false;
      }
    }
    return true;
  };
  const Order8 order{U, a.lag, a.behind};

  constexpr uint32_t idesc1 = idesc_f16(128, N, false, false);
  constexpr uint32_t idesc2 = idesc_f16(128, N, true, false);

  const int sb = a.seg_ptr[cluster_id], se = a.seg_ptr[cluster_id + 1];
  const bool converter = warp < 4 || (warp >= 8 && warp < 12);
  // the converters read only the codes; the other roles wait for the kernel before
  if (!converter) after_previous();
  if (sb >= se) {
    // no rows: straight to the teardown
  } else if (converter) {
    // -------------------------------------------------------------- converters: codes -> FP16 operand
    // thread: 16 codes at (lane & 3) of either 64-column chunk, rows 8 (warp mod 4) +
    // (lane >> 2) + 32 i; eight lanes write two rows of four 16-byte pieces, all eight
    // bank groups
    const uint32_t grp = warp < 4 ? 0 : 1;
    const int row0 = 8 * (warp & 3) + (lane >> 2);
    const uint32_t at0 = row0 * 128 + (((2 * (lane & 3)) ^ (lane >> 2)) << 4);
    const uint32_t at1 = row0 * 128 + (((2 * (lane & 3) + 1) ^ (lane >> 2)) << 4);
    const uint64_t pol = grp == 0 || !a.hints ? l2_policy_evict_last() : l2_policy_evict_first();
    uint4 buf[kDepth][8];
    uint32_t unit[kDepth];  // the unit in buf[x]; ~0: none left
    Run8 run = run_at(a.segs, sb, se);
    uint32_t base_g = 0;  // units before the run
    int t = 0, u = 0;
    bool more = true;
    // the next unit of this group's pass into v
    auto fetch = [&](uint4 (&v)[8]) -> uint32_t {
      if (!more) return ~0u;
      const uint32_t g = base_g + (grp == 0 ? order.first(t, u, run.ntiles) : order.second(t, u, run.ntiles));
      const int64_t r0 = run.row0 + static_cast<int64_t>(t) * kBM + row0;
      const int c = c0 + 128 * u + 16 * (lane & 3);
      const unsigned char* p = a.codes + r0 * a.ld + c;
      const int64_t step = 32 * a.ld;
      if (r0 - row0 + kBM <= a.n && c0 + 128 * (u + 1) <= a.ld) {  // the whole unit lies in the matrix
#pragma unroll
        for (int i = 0; i < 8; i += 2, p += step) {
          v[i] = ld_codes(p, pol);
          v[i + 1] = ld_codes(p + 64, pol);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          v[i] = c + 64 * (i & 1) < a.ld && r0 + 32 * (i >> 1) < a.n ? ld_codes(p + (i >> 1) * step + 64 * (i & 1), pol)
                                                                   : make_uint4(0u, 0u, 0u, 0u);
      }
      if (++u == U) {
        u = 0;
        if (++t == run.ntiles) {
          t = 0;
          base_g += 2u * static_cast<uint32_t>(run.ntiles) * static_cast<uint32_t>(U);
          more = run.sj < se;
          if (more) run = run_at(a.segs, run.sj, se);
        }
      }
      return g;
    };
#pragma unroll
    for (int x = 0; x < kDepth; ++x) unit[x] = fetch(buf[x]);
    Place8 at;
    bool ok = true;
    while (ok && unit[0] != ~0u) {
#pragma unroll
      for (int x = 0; x < kDepth; ++x) {
        if (!ok || unit[x] == ~0u) continue;
        at.to(unit[x], R);
        if (!(ok = wait_fills(at.slot, at.fill) &&
                   wait(S_RING0 + kMaxRing + static_cast<int>(at.slot), (at.fill & 1) ^ 1, false)))
          continue;
        __syncwarp();
        if ((warp & 3) == 0 && lane == 0) fills[at.slot] = at.fill + 1;
        unsigned char* dst = sRing + at.slot * kUnitBytes;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 v = buf[x][i];
          uint4 h0, h1;
          e4m3x4_to_f16x4(v.x, h0.x, h0.y);
          e4m3x4_to_f16x4(v.y, h0.z, h0.w);
          e4m3x4_to_f16x4(v.z, h1.x, h1.y);
          e4m3x4_to_f16x4(v.w, h1.z, h1.w);
          unsigned char* q = dst + (i & 1) * kChunkBytes + (i >> 1) * 32 * 128;
          *reinterpret_cast<uint4*>(q + at0) = h0;
          *reinterpret_cast<uint4*>(q + at1) = h1;
        }
        fence_async_smem();  // the MMAs read these tiles through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[S_RING0 + at.slot]);
        unit[x] = fetch(buf[x]);
      }
    }
  } else {
    // -------------------------------------------------------------- issuers and epilogue, run by run
    const int ot = warp < 8 ? tid - 128 : tid - 384 + 128;  // 0 .. kOthers8 - 1
    uint32_t T = 0, pieces = 0, epi_phase = 0;
    uint32_t base_g = 0;  // units before the run
    Place8 at;
    for (int si = sb; si < se;) {
      const Run8 run = run_at(a.segs, si, se);
      __syncwarp();
      // every role finished the previous run; all leave together after an abort
      if (bar_or(1, kOthers8, *abort_flag != 0)) break;
      // this slice of Z as [Z_hi | Z_lo]^T in FP16 (N rows x DC, K-major, SWIZZLE_128B)
      if (si == sb || a.z_stride != 0)
        stage_z<K, F16Op>(sB1, a.Z + a.z_stride * a.segs[si].part, c0, DC, a.d, ot, kOthers8);
      fence_async_smem();
      bar_sync(1, kOthers8);

      if (warp >= kIssue1) {
        if (lane == 0) {
          // ---------------------------------------------------------- MMA issuers (one per pass)
          bool ok = true;
          auto ready = [&](uint32_t g) -> bool {
            at.to(base_g + g, R);
            return wait_fills(at.slot, at.fill + 1) && wait(S_RING0 + static_cast<int>(at.slot), at.fill & 1, false);
          };
          if (warp == kIssue1) {
            const uint32_t bS = su32(sB1);
            uint32_t buf = T % ND1, use = T / ND1;
            for (int t = 0; ok && t < run.ntiles; ++t) {
              if (!(ok = wait(S_D1EMPTY0 + static_cast<int>(buf), (use + 1) & 1, false))) break;
              for (int u = 0; u < U; ++u) {
                if (!(ok = ready(order.first(t, u, run.ntiles)))) break;
                tc_fence_after();
                const uint32_t aS = su32(sRing + at.slot * kUnitBytes);
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                  for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t ad = sdesc(aS + j * kChunkBytes + kk * 32, 16, 1024);
                    const uint64_t bd = sdesc(bS + (2 * u + j) * N * 128 + kk * 32, 16, 1024);
                    mma_bf16(tmem + buf * N, ad, bd, idesc1, (u | j | kk) != 0);
                  }
                mma_commit(&bar[S_RING0 + kMaxRing + at.slot]);
              }
              if (ok) mma_commit(&bar[S_D1FULL0 + buf]);
              if (++buf == static_cast<uint32_t>(ND1)) {
                buf = 0;
                ++use;
              }
            }
          } else {
            for (int t = 0; ok && t < run.ntiles; ++t) {
              const uint32_t Tg = T + t, buf = Tg & 1;
              if (!(ok = wait(S_B2FULL0 + static_cast<int>(buf), (Tg >> 1) & 1, false))) break;
              // a new piece accumulates from zero: the previous one's sums have been read out
              if (t % TP == 0 && !(ok = wait(S_D2EMPTY, (pieces + t / TP + 1) & 1, false))) break;
              const uint32_t bS = su32(sB2 + buf * B2BUF);
              for (int u = 0; u < U; ++u) {
                if (!(ok = ready(order.second(t, u, run.ntiles)))) break;
                tc_fence_after();
                const uint32_t aS = su32(sRing + at.slot * kUnitBytes);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                  const uint64_t ad = sdesc(aS + kk * 2048, kChunkBytes, 1024);
                  const uint64_t bd = sdesc(bS + (kk >> 2) * N * 128 + (kk & 3) * 32, 16, 1024);
                  mma_bf16(tD2 + u * N, ad, bd, idesc2, (t % TP == 0 && kk == 0) ? 0u : 1u);
                }
                mma_commit(&bar[S_RING0 + kMaxRing + at.slot]);
              }
              if (!ok) break;
              mma_commit(&bar[S_B2FREE0 + buf]);
              if (t % TP == TP - 1 || t == run.ntiles - 1) mma_commit(&bar[S_D2FULL]);
            }
          }
          // the first pass's last D1 is full before the second pass ends, and the epilogue
          // waits for that, so Z is free when the run is over
        }
      } else {
        // ------------------------------------------------------------ epilogue
        const int r = (warp - 4) * 32 + lane;
        const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
        bool ok = true;
        auto epi_sync = [&]() -> bool {
          mbar_arrive(&bar[S_EPI]);
          return wait(S_EPI, (epi_phase++) & 1, false);
        };
        // Y slice = S (D2[:, :K] + D2[:, K:]) of piece `piece` -> P[slot]
        auto drain = [&](int piece) -> bool {
          if (!wait(S_D2FULL, (pieces + piece) & 1, false)) return false;
          tc_fence_after();
          float* Pd = a.P + static_cast<int64_t>(a.segs[si + piece].slot) * a.d * K;
          for (int b = 0; b < U; ++b) {
            float y[K];
#pragma unroll
            for (int q = 0; q < N / 16; ++q) {
              float v[16];
              tmem_ld16(tD2 + lane_base + b * N + q * 16, v);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int col = q * 16 + i;
                if (col < K) y[col] = v[i];
                else y[col - K] += v[i];
              }
            }
            const int dcol = c0 + b * 128 + (warp & 3) * 32 + lane;
            if (dcol < a.d) {
              float4* dst = reinterpret_cast<float4*>(Pd + static_cast<int64_t>(dcol) * K);
#pragma unroll
              for (int j = 0; j < K; j += 4)
                dst[j / 4] = make_float4(a.smax2 * y[j], a.smax2 * y[j + 1], a.smax2 * y[j + 2], a.smax2 * y[j + 3]);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar[S_D2EMPTY]);
          return true;
        };
        for (int t = 0; ok && t < run.ntiles; ++t) {
          const uint32_t Tg = T + t, buf = Tg % ND1, wb = Tg & 1;
          if (!(ok = wait(S_D1FULL0 + static_cast<int>(buf), (Tg / ND1) & 1, false))) break;
          tc_fence_after();
          float w[K];
#pragma unroll
          for (int q = 0; q < N / 16; ++q) {
            float v[16];
            tmem_ld16(tmem + lane_base + buf * N + q * 16, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int col = q * 16 + i;
              if (col < K) w[col] = v[i];
              else w[col - K] += v[i];
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar[S_D1EMPTY0 + buf]);
          const int64_t grow = run.row0 + static_cast<int64_t>(t) * kBM + r;
          const bool valid = grow < run.row1;
          const float sc = valid ? a.scales[grow] : 0.f;
          if (!valid) {
#pragma unroll
            for (int j = 0; j < K; ++j) w[j] = 0.f;
          }
          if (CL > 1 &&
              !(ok = sum_over_cluster<K>(
                    w, r, crank, CL, RPC, sW, sWrecv, &bar[S_REDFULL], &bar[S_WFULL], [&] { return wait(S_REDFULL, Tg & 1, true); },
                    [&] { return wait(S_WFULL, Tg & 1, true); }, epi_sync)))
            break;
          // row scale: W_r <- W_r s_r^2 / S (so the FP16 operand cannot overflow)
          const float f = sc * sc / a.smax2;
#pragma unroll
          for (int j = 0; j < K; ++j) w[j] *= f;
          if (!(ok = wait(S_B2FREE0 + static_cast<int>(wb), ((Tg >> 1) + 1) & 1, false))) break;
          unsigned char* B2 = sB2 + wb * B2BUF;
#pragma unroll
          for (int j = 0; j < K; ++j) {
            const uint16_t hi = f16_bits(w[j]);
            const uint16_t lo = f16_bits(w[j] - f16_val(hi));
            *reinterpret_cast<uint16_t*>(B2 + sw128_off(j, r, N)) = hi;
            *reinterpret_cast<uint16_t*>(B2 + sw128_off(K + j, r, N)) = lo;
          }
          fence_async_smem();
          mbar_arrive(&bar[S_B2FULL0 + wb]);
          if (t % TP == TP - 1 || t == run.ntiles - 1) ok = drain(t / TP);
        }
      }
      T += run.ntiles;
      pieces += (run.ntiles + TP - 1) / TP;
      base_g += 2u * static_cast<uint32_t>(run.ntiles) * static_cast<uint32_t>(U);
      si = run.sj;
    }
  }

  before_next();
  if (tid == 4 * 32) bulk_wait_read0();  // the epilogue's last copies have read shared memory
  // ---- teardown: MMAs retired, no remote traffic, then free TMEM
  if (warp >= kIssue1 && lane == 0) mma_commit(&bar[S_DONE]);
  __syncthreads();
  if (warp == 0) {
    const uint32_t addr = su32(&bar[S_DONE]);
    const long long t0 = clock64();
    while (!mbar_try(addr, 0) && clock64() - t0 < kTimeoutCycles) {
    }
  }
  __syncthreads();
  cluster_sync_all();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
}

template <int K>
cudaLaunchConfig_t tcs8_config(unsigned grid, int cl, size_t smem, cudaStream_t s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kThreads8, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cl);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int K>
int tcs8_active_clusters(int cl, size_t smem) {
  if (allow_max_dynamic_smem(reinterpret_cast<const void*>(step_tcs8_kernel<K>)) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = tcs8_config<K>(static_cast<unsigned>(cl), cl, smem, nullptr, attr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, step_tcs8_kernel<K>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

template <int K>
cudaError_t launch_tcs8_t(const TcsPlan& p, const Tcs8Args& a, Lane at) {
  cudaError_t e = allow_max_dynamic_smem(reinterpret_cast<const void*>(step_tcs8_kernel<K>));
  if (e != cudaSuccess) return e;
  return launch_on(at, step_tcs8_kernel<K>, dim3(static_cast<unsigned>(p.nclusters * p.cluster)), kThreads8, p.smem,
                   static_cast<unsigned>(p.cluster), a);
}

}  // namespace

namespace {
bool tcs8_plan_slice(int d, int k, int sms, const TcsTuning& tune, int ncd_max, TcsPlan* p);
}  // namespace

// Without a slice width from the tuning, the widest slice that has a plan (fewest
// CTAs per cluster, least W exchange).
bool tcs8_plan(int d, int k, int sms, const TcsTuning& tune, TcsPlan* p) {
  const int K = k <= 8 ? 8 : (k <= 16 ? 16 : 32);
  if (tune.slice_cols >= 128) return tcs8_plan_slice(d, k, sms, tune, (tune.slice_cols / 128) * 2, p);
  for (int ncd_max = K == 32 ? 8 : 16; ncd_max >= 4; ncd_max /= 2)
    if (tcs8_plan_slice(d, k, sms, tune, ncd_max, p)) return true;
  return false;
}

namespace {
bool tcs8_plan_slice(int d, int k, int sms, const TcsTuning& tune, int ncd_max, TcsPlan* p) {
  const int K = k <= 8 ? 8 : (k <= 16 ? 16 : 32);
  const int N = 2 * K;
  int nc = (d + 63) / 64;
  nc += nc & 1;
  int cl = 1;
  while (cl * ncd_max < nc) cl *= 2;
  if (cl > 8) return false;
  int ncd = (nc + cl - 1) / cl;
  ncd += ncd & 1;
  const uint32_t B1 = static_cast<uint32_t>(ncd) * N * 128;
  const uint32_t B2 = 2u * (2u * N * 128);
  const uint32_t W = cl > 1 ? 128u * K * 4 : 0u;
  const uint32_t bars = kNumBars8 * 8 + 16 + kMaxRing * 4;  // barriers, TMEM holder, abort flag, fills
  const int avail = kSmemLimit - 1024 - static_cast<int>(B1 + B2 + 2 * W + bars);
  // operand ring of 32 KB units: three at least (the narrower slices' plans start there), up
  // to four (the converters' registers hold the units in flight, the ring only what
  // the MMAs read)
  int ring = avail / kUnitBytes;
  if (ring < 3 || tune.ring_units == 1) return false;
  if (ring > 4) ring = 4;
  if (tune.ring_units > 0 && ring > tune.ring_units) ring = tune.ring_units;
  p->K = K;
  p->planes = 1;
  p->ncd = ncd;
  p->cluster = cl;
  p->ring = ring;
  const int lag = tune.lag_units > 0 ? tune.lag_units : tcs8_default_lag(cl);
  const int U = ncd / 2;
  p->lag = lag < U ? lag : U;
  p->prefetch = 0;
  p->hints = 1;  // first pass evict_last, second pass evict_first
  p->off_B1 = static_cast<uint32_t>(ring) * kUnitBytes;
  p->off_B2 = p->off_B1 + B1;
  p->off_W = p->off_B2 + B2;
  p->off_Wrecv = p->off_W + W;
  p->off_bar = p->off_Wrecv + W;
  p->smem = p->off_bar + bars + 1024;
  // a second tile between the passes where W crosses a cluster and tensor memory holds
  // three D1
  p->behind = cl > 1 && 3 * N + U * N <= 512 ? 2 : 1;
  const uint32_t used = static_cast<uint32_t>((p->behind + 1) * N + U * N);
  uint32_t cols = 32;
  while (cols < used) cols *= 2;
  if (cols > 512) return false;
  p->tmem_cols = cols;
  if (p->smem > static_cast<size_t>(kSmemLimit)) return false;
  const int active = K == 8 ? tcs8_active_clusters<8>(cl, p->smem)
                            : K == 16 ? tcs8_active_clusters<16>(cl, p->smem) : tcs8_active_clusters<32>(cl, p->smem);
  p->nclusters = sms / cl;
  if (active > 0 && active < p->nclusters) p->nclusters = active;
  p->fp8 = 1;
  return p->nclusters >= 1;
}
}  // namespace

cudaError_t launch_step_tcs8(const TcsPlan& p, const void* codes, int64_t n, int64_t ld, const Segment* segs,
                             const int* seg_ptr, const float* Z, int64_t z_stride, float* P, int d, const float* scales,
                             float smax2, int* status, Lane at) {
  Tcs8Args a;
  a.codes = static_cast<const unsigned char*>(codes);
  a.n = n;
  a.ld = ld;
  a.segs = segs;
  a.seg_ptr = seg_ptr;
  a.Z = Z;
  a.z_stride = z_stride;
  a.P = P;
  a.d = d;
  a.status = status;
  a.scales = scales;
  a.smax2 = smax2;
  a.ncd = p.ncd;
  a.ring = p.ring;
  a.lag = p.lag;
  a.behind = p.behind;
  a.hints = p.hints;
  a.off_B1 = p.off_B1;
  a.off_B2 = p.off_B2;
  a.off_W = p.off_W;
  a.off_Wrecv = p.off_Wrecv;
  a.off_bar = p.off_bar;
  a.tmem_cols = p.tmem_cols;
  if (p.K == 8) return launch_tcs8_t<8>(p, a, at);
  if (p.K == 16) return launch_tcs8_t<16>(p, a, at);
  return launch_tcs8_t<32>(p, a, at);
}

}  // namespace lp

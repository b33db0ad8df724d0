// What the attention sublayer adds to the residual stream (Sec. 3), on the tensor cores:
//   residual update:   y = x + O W_o^T                 (bf16 in and out, fp32 accumulation)
//   token-level drift: drift[b] = sum_{t in block b} ||W_o (O_a[t] - O_b[t])||^2
// O is [N, K] with K = H * 64 (the concatenated head outputs), W_o is [d_model, K] (Linear
// weight, out x in), x and y are [N, d_model].
//
// One tile = 256 tokens x 256 output channels of a CTA pair (cta_group::2: M256 N256 K16, each
// CTA holding 128 of A's rows, 128 of B's rows and 128 rows of the accumulator), reduced over K
// in 64-wide slices through a TMA ring (128-byte swizzle, both operands K-major).  What bounds
// the kernel is operand delivery into the SM (about 50 bytes per cycle): a pair brings 32 KB per
// SM and slice for the 128 x 256 x 64 products of one CTA, where a CTA by itself needs 48 KB
// (43,968 tokens, K = d_model = 1024: 86.9 us with single CTAs, 78.5 with pairs, 74.2 with the
// epilogue on eight warps instead of four; 1.24 PFLOP/s, and the tensor pipe's clock under its
// power limit is the next bound: with half of every load left out it still took 62 us).  Per CTA 320 threads:
//   warp 0     TMA of its half of the O and W_o slices (the drift variant loads O_a and O_b
//              slices); the bytes of both CTAs are counted by the barrier of the rank-0 CTA;
//   warp 1     TMEM owner; in the rank-0 CTA one elected lane of the converged warp issues per
//              slice 4 MMAs for the pair (the drift variant: 4 into each of two accumulators);
//   warps 2-9  epilogue, row r = TMEM lane, four warps per half of the channels: residual update: the tile's x (loaded by TMA into
//              a swizzled staging area) plus the accumulator, rounded to bf16 in place and
//              written out by TMA bulk stores; drift: the squared difference of the two
//              accumulators summed over the row's channels, then over each block's 64 rows
//              in a fixed order.
// The residual update runs persistent pairs over the tiles with two TMEM accumulators, so a
// tile's epilogue overlaps the next tile's MMAs; the drift variant gives each 256-token stripe
// to a cluster of one, two or four pairs, which take its channel tiles in turn and add up
// their rows' sums through distributed shared memory.
// Every mbarrier wait is bounded; a wait that gives up records RESS_ETIMEOUT, makes the CTA
// leave its loops (and, as its waits run out, the other one), lets copies and MMAs already
// issued finish (again bounded); the pair then meets at a cluster barrier, frees TMEM and
// returns.

#include <cudaTypedefs.h>

#include "ress_internal.cuh"
#include "sm100_ptx.cuh"

namespace ress {
using namespace ptx;

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();

namespace {

constexpr int kOThreads = 320;
constexpr int kOM = 128;                      // tokens per tile and CTA
constexpr int kON = 256;                      // output channels per tile
constexpr uint32_t kABytes = kOM * 128;       // 128 x 64 bf16
constexpr uint32_t kBBytes = kON / 2 * 128;   // 128 x 64 bf16: this CTA's half of B's rows
constexpr uint32_t kOCols = 512;              // TMEM: two 128 x 256 fp32 accumulators
constexpr uint64_t kOWaitNs = 2000000000ull;  // 2 s per wait
constexpr uint64_t kODrainNs = 200000000ull;  // 0.2 s to drain after an abort

enum { kResidual = 0, kDrift = 1 };

// Shared-memory layout.  Residual: five stages of A | B, then X (4 boxes of 128 x 64 bf16).
// Drift: four stages of A | A2 | B.
template <int MODE>
constexpr int kOStages = MODE == kDrift ? 4 : 5;
template <int MODE>
constexpr uint32_t kStageBytes = (MODE == kDrift ? 2 : 1) * kABytes + kBBytes;
constexpr uint32_t kOffX = kOStages<kResidual> * kStageBytes<kResidual>;
constexpr uint32_t kOData = kOffX + 4 * 16384;  // the larger of the two layouts
static_assert(kOStages<kDrift> * kStageBytes<kDrift> <= kOData, "drift layout fits the residual one");

struct OCtl {
  float rowsum[2][kOM];
  float blocksum[4];
  uint64_t full[5], empty[5], acc_full[2], acc_empty[2], x_full[2];
  uint32_t tmem_base;
  int abort;
};

struct OParams {
  int N, K, Dm, nb;
  int mtiles, ntiles;  // tiles of 256 tokens, of 256 channels
  // residual: the first `whole` tiles run whole; each one after them as `parts` units of
  // 256 / parts channels
  int whole, parts;
  int group;  // drift: pairs per stripe (cluster of 2 group CTAs), at most ntiles
  bool has_x;
  float* drift;
  uint32_t* status;
};

__device__ __forceinline__ bool o_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort, kOWaitNs) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}

__device__ __forceinline__ void o_give_up(OCtl& C, uint32_t* status) {
  flag_status(status, kStatusTimeout);
  *reinterpret_cast<volatile int*>(&C.abort) = 1;
}

// Named barriers of the four epilogue warps of channel half hf (0 or 1); the first also ANDs
// a flag across them.
__device__ __forceinline__ bool o_epi_sync_and(int hf, bool v) {
  __syncwarp();
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "r"(1 + hf)
      : "memory");
  return r != 0;
}
// The same of all eight epilogue warps (drift).
__device__ __forceinline__ bool o_epi_sync_and_all(bool v) {
  __syncwarp();
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 5, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void o_epi_sync_all() {
  __syncwarp();
  asm volatile("bar.sync 5, 256;" ::: "memory");
}
__device__ __forceinline__ void o_epi_sync(int hf) {
  __syncwarp();
  asm volatile("bar.sync %0, 128;" ::"r"(3 + hf) : "memory");
}

// One unit of work: rows of stripe mt, channels [col, col + width).
struct OUnit {
  int mt, col, width;
};
// Drift: persistent pairs over whole stripes, or a cluster of p.group pairs per stripe, which take
// its channel tiles in turn.
template <int MODE>
__device__ __forceinline__ int units_of_pair(const OParams& p) {
  if (MODE == kDrift && p.group == 1)
    return ((p.mtiles - 1 - (int)(blockIdx.x >> 1)) / (int)(gridDim.x >> 1) + 1) * p.ntiles;
  if (MODE == kDrift) return (p.ntiles - 1 - (int)(cluster_rank() >> 1)) / p.group + 1;
  const int units = p.whole + (p.mtiles * p.ntiles - p.whole) * p.parts;
  return (units - 1 - (int)(blockIdx.x >> 1)) / (int)(gridDim.x >> 1) + 1;
}
template <int MODE>
__device__ __forceinline__ OUnit unit_of_pair(const OParams& p, int k) {
  if (MODE == kDrift && p.group == 1)
    return OUnit{(int)(blockIdx.x >> 1) + k / p.ntiles * (int)(gridDim.x >> 1), kON * (k % p.ntiles), kON};
  if (MODE == kDrift)
    return OUnit{(int)blockIdx.x / (2 * p.group), kON * ((int)(cluster_rank() >> 1) + k * p.group), kON};
  // consecutive tiles share their token stripe, so O slices are re-read from L2
  const int u = (int)(blockIdx.x >> 1) + k * (int)(gridDim.x >> 1);
  if (u < p.whole) return OUnit{u / p.ntiles, kON * (u % p.ntiles), kON};
  const int t = p.whole + (u - p.whole) / p.parts, w = kON / p.parts;
  return OUnit{t / p.ntiles, kON * (t % p.ntiles) + w * ((u - p.whole) % p.parts), w};
}

template <int MODE>
__global__ void __launch_bounds__(kOThreads, 1)
    k_oproj(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmA2,
            const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmBpart,
            const __grid_constant__ CUtensorMap tmX,
            const __grid_constant__ CUtensorMap tmY, const OParams p) {
  const int nunits = units_of_pair<MODE>(p);  // at least 1: at most one pair per unit
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  OCtl& C = *reinterpret_cast<OCtl*>(base + kOData);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &C.abort;
  const int ksteps = p.K / 64;
  constexpr int kStages = kOStages<MODE>;
  const int rank = (int)cluster_rank() & 1;   // this CTA's half of the pair's rows
  const int lead = (int)cluster_rank() & ~1;  // the pair's rank-0 CTA
  const uint32_t both = 3u << lead;
  auto A = [&](int s) { return base + s * kStageBytes<MODE>; };
  auto A2 = [&](int s) { return A(s) + kABytes; };
  auto B = [&](int s) { return A(s) + (MODE == kDrift ? 2 : 1) * kABytes; };
  uint8_t* X = base + kOffX;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&C.full[s], 1);
      mbar_init(&C.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&C.acc_full[b], 1);
      mbar_init(&C.acc_empty[b], 16);  // the epilogue warps of both CTAs
      mbar_init(&C.x_full[b], 1);
    }
    C.abort = 0;
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
    if (MODE == kDrift) prefetch_tensormap(&tmA2);
    if (MODE == kResidual) {
      prefetch_tensormap(&tmY);
      if (p.has_x) prefetch_tensormap(&tmX);
    }
  }
  if (warp == 1) tmem_alloc_pair(&C.tmem_base, kOCols);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist
  tc_fence_after();
  const uint32_t tmem = C.tmem_base;
  pdl_wait();

  if (warp == 0) {
    // ================================ loads ==========================================
    // the barriers of the rank-0 CTA count the bytes of both
    int it = 0;
    bool failed = false;
    for (int k = 0; k < nunits && !failed; ++k) {
      const OUnit t = unit_of_pair<MODE>(p, k);
      // the stripe of the pair's next unit into L2 while this one runs (by the pair that takes
      // the stripe's first channels): 69.4 -> 67.4 us at 43,968 tokens, warm inputs
      const OUnit t2 = unit_of_pair<MODE>(p, min(k + 1, nunits - 1));
      const bool ahead = MODE == kResidual && k + 1 < nunits && t2.col == 0;
      for (int ks = 0; ks < ksteps; ++ks, ++it) {
        const int s = it % kStages, u = it / kStages;
        if (u > 0 && !o_wait(&C.empty[s], (u - 1) & 1, abort)) {
          failed = true;
          break;
        }
        if (lane == 0) {
          const uint32_t bytes = (MODE == kDrift ? 2 : 1) * kABytes + t.width / 2 * 128;
          if (rank == 0) mbar_arrive_expect_tx(&C.full[s], 2 * bytes);
          const uint32_t full = cluster_addr(&C.full[s], lead);
          const int row = kOM * (2 * t.mt + rank);
          tma_load_3d_pair(A(s), &tmA, full, 64 * ks, row, 0);
          if (MODE == kDrift) tma_load_3d_pair(A2(s), &tmA2, full, 64 * ks, row, 0);
          tma_load_3d_pair(B(s), t.width == kON ? &tmB : &tmBpart, full, 64 * ks,
                           t.col + t.width / 2 * rank, 0);
          if (ahead) tma_prefetch_3d(&tmA, 64 * ks, kOM * (2 * t2.mt + rank), 0);
        }
        __syncwarp();
      }
    }
    pdl_trigger();  // every slice of the CTA's tiles is on its way
    // the pair's MMAs release every stage in both CTAs: nothing arrives here after the end
    for (int q = max(0, it - kStages); q < it && !failed; ++q)
      if (!o_wait(&C.empty[q % kStages], (q / kStages) & 1, abort)) failed = true;
    if (failed && lane == 0) {
      o_give_up(C, p.status);
      volatile int no_abort = 0;  // copies already issued land before the memory goes away (the
      // rank-1 CTA's are counted in the other one: its waits here just run out)
      for (int q = max(0, it - kStages); q < it; ++q)
        mbar_wait(&C.full[q % kStages], (q / kStages) & 1, &no_abort, kODrainNs);
    }
    __syncwarp();
  } else if (warp == 1 && rank == 1) {
    // the rank-0 CTA issues the pair's MMAs
  } else if (warp == 1) {
    // ================================ MMAs ===========================================
    const bool leader = elect_one();
    int it = 0;
    bool failed = false;
    if (__popc(__ballot_sync(0xffffffffu, leader)) != 1) {  // exactly one issuing lane
      if (lane == 0) {
        flag_status(p.status, kStatusBadRow);
        *abort = 1;
      }
      failed = true;
    }
    for (int k = 0; k < nunits && !failed; ++k) {
      const uint32_t idesc = idesc_bf16_f32(2 * kOM, unit_of_pair<MODE>(p, k).width, false);
      const int b = MODE == kDrift ? 0 : (k & 1);
      const int use = MODE == kDrift ? k : (k >> 1);  // earlier uses of accumulator b
      if (use > 0 && !o_wait(&C.acc_empty[b], (use - 1) & 1, abort)) {
        failed = true;
        break;
      }
      tc_fence_after();
      const uint32_t acc = tmem + (MODE == kDrift ? 0u : (uint32_t)kON * b);
      for (int ks = 0; ks < ksteps; ++ks, ++it) {
        const int s = it % kStages;
        if (!o_wait(&C.full[s], (it / kStages) & 1, abort)) {
          failed = true;
          break;
        }
        tc_fence_after();
        if (leader) {
          const uint32_t a = smem_u32(A(s)), bb = smem_u32(B(s));
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_bf16_ss_pair(acc, sdesc_sw128(a + 32 * kk), sdesc_sw128(bb + 32 * kk), idesc,
                        (ks > 0 || kk > 0) ? 1u : 0u);
          if (MODE == kDrift) {
            const uint32_t a2 = smem_u32(A2(s));
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_bf16_ss_pair(tmem + kON, sdesc_sw128(a2 + 32 * kk), sdesc_sw128(bb + 32 * kk), idesc,
                          (ks > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit_pair(&C.empty[s], both);
          if (ks + 1 == ksteps) mma_commit_pair(&C.acc_full[b], both);
        }
        __syncwarp();
      }
    }
    if (failed && lane == 0) {
      o_give_up(C, p.status);
      if (it > 0) {  // MMAs still running must finish before TMEM is freed
        volatile int no_abort = 0;
        const int q = it - 1;
        mbar_wait(&C.empty[q % kStages], (q / kStages) & 1, &no_abort, kODrainNs);
      }
    }
    __syncwarp();
  } else {
    // ================================ epilogue =======================================
    // two groups of four warps, each a half of the tile's channels with its own staging
    // boxes, x barrier and stores
    const int hf = (warp - 2) >> 2;
    const int quarter = warp & 3;
    const int r = 32 * quarter + lane;  // row of the tile = TMEM lane
    const uint32_t lane_base = ((uint32_t)(32 * quarter) << 16) + kON / 2 * hf;
    const bool leader = (warp - 2) % 4 == 0 && lane == 0;
    uint8_t* Xh = X + 2 * hf * 16384;
    float rowsum = 0.f;
    // 64-channel boxes of this half in a unit (a part of a tile may have none)
    auto boxes_of = [&](const OUnit& t) { return max(0, min(2, t.width / 64 - 2 * hf)); };
    auto load_x = [&](int k) {  // this half of unit k's x into the staging boxes
      const OUnit t = unit_of_pair<MODE>(p, k);
      const int boxes = boxes_of(t);
      if (boxes == 0) return;
      mbar_arrive_expect_tx(&C.x_full[hf], boxes * 16384);
      for (int q = 0; q < boxes; ++q)
        tma_load_3d(Xh + q * 16384, &tmX, &C.x_full[hf], t.col + kON / 2 * hf + 64 * q,
                    kOM * (2 * t.mt + rank), 0);
    };
    if (MODE == kResidual && p.has_x && leader) load_x(0);
    for (int k = 0; k < nunits; ++k) {
      const OUnit t = unit_of_pair<MODE>(p, k);
      const int boxes = boxes_of(t);
      const int row0 = kOM * (2 * t.mt + rank), col0 = t.col + kON / 2 * hf;
      const int b = MODE == kDrift ? 0 : (k & 1);
      const int use = MODE == kDrift ? k : (k >> 1);
      if (MODE == kResidual && p.has_x && leader && k + 1 < nunits) {  // the next unit's x into L2
        const OUnit t2 = unit_of_pair<MODE>(p, k + 1);
        for (int q = 0; q < boxes_of(t2); ++q)
          tma_prefetch_3d(&tmX, t2.col + kON / 2 * hf + 64 * q, kOM * (2 * t2.mt + rank), 0);
      }
      bool ok = o_wait(&C.acc_full[b], use & 1, abort);
      if (MODE == kResidual && p.has_x && ok && boxes > 0) ok = o_wait(&C.x_full[hf], k & 1, abort);
      if (!(MODE == kDrift ? o_epi_sync_and_all(ok) : o_epi_sync_and(hf, ok))) {  // all leave together
        if (!ok && lane == 0) o_give_up(C, p.status);
        break;
      }
      tc_fence_after();
      if (MODE == kDrift) {
#pragma unroll 1
        for (int q = 0; q < kON / 64; ++q) {
          uint32_t va[32], vb[32];
          RESS_TMEM_LD32(tmem + lane_base + 32 * q, va);
          RESS_TMEM_LD32(tmem + kON + lane_base + 32 * q, vb);
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float d = __uint_as_float(va[e]) - __uint_as_float(vb[e]);
            rowsum = fmaf(d, d, rowsum);
          }
        }
      } else {
        const uint32_t acc = tmem + (uint32_t)kON * b + lane_base;
#pragma unroll 1
        for (int q = 0; q < 2 * boxes; ++q) {  // channels 32q .. 32q + 31: box q/2, chunks 4(q%2)..
          uint32_t v[32];
          RESS_TMEM_LD32(acc + 32 * q, v);
          uint8_t* row = Xh + (q >> 1) * 16384 + r * 128;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint4* at = reinterpret_cast<uint4*>(row + (((4 * (q & 1) + c) ^ (r & 7)) << 4));
            uint4 xv = make_uint4(0u, 0u, 0u, 0u);
            if (p.has_x) xv = *at;
            const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
            uint32_t yw[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              yw[e] = cvt_bf16x2(__uint_as_float(v[8 * c + 2 * e]) + bf16_lo(xw[e]),
                                 __uint_as_float(v[8 * c + 2 * e + 1]) + bf16_hi(xw[e]));
            *at = make_uint4(yw[0], yw[1], yw[2], yw[3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_addr(&C.acc_empty[b], lead));  // may be reused
      if (MODE == kDrift && p.group == 1 && (k + 1) % p.ntiles == 0) {
        // the stripe is complete: rows over their channel halves, 64-token blocks over their rows,
        // warp tree by warp tree (as after a cluster's tiles, below)
        C.rowsum[hf][r] = rowsum;
        rowsum = 0.f;
        o_epi_sync_all();
        if (hf == 0) {
          float v = 0.f;
#pragma unroll
          for (int q = 0; q < 2; ++q) v += C.rowsum[q][r];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) C.blocksum[quarter] = v;
        }
        o_epi_sync_all();
        const int blk = 2 * (2 * t.mt + rank) + (quarter >> 1);
        if (hf == 0 && lane == 0 && (quarter & 1) == 0 && blk < p.nb && !*abort)
          p.drift[blk] = C.blocksum[quarter] + C.blocksum[quarter + 1];
      }
      if (MODE == kResidual) {
        fence_proxy_async_smem();
        o_epi_sync(hf);
        if (leader) {
#pragma unroll 1
          for (int q = 0; q < boxes; ++q)
            if (col0 + 64 * q < p.Dm && row0 < p.N)
              tma_store_3d(&tmY, Xh + q * 16384, col0 + 64 * q, row0, 0);
          bulk_commit();
          bulk_wait_read_all();  // the staging boxes are free again
          if (p.has_x && k + 1 < nunits) load_x(k + 1);
        }
      }
    }
    if (MODE == kDrift && p.group > 1) C.rowsum[hf][r] = rowsum;
    if (leader) bulk_wait_read_all();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the pair's MMAs and barrier arrivals are over in both CTAs
  if (MODE == kDrift && p.group > 1) {
    // the cluster's first pair sums its rows over the pairs (and their channel halves) in
    // order, then each 64-token block over its rows, warp tree by warp tree
    if (cluster_rank() < 2 && threadIdx.x < kOM) {
      float v = 0.f;
      for (int g = 0; g < p.group; ++g)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
          v += ld_cluster_f32(cluster_addr(&C.rowsum[hf][threadIdx.x], 2 * g + rank));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) C.blocksum[warp] = v;
    }
    cluster_sync();  // the other CTAs' sums have been read
    if (cluster_rank() < 2 && threadIdx.x < 2) {
      const int blk = 2 * (2 * ((int)blockIdx.x / (2 * p.group)) + rank) + (int)threadIdx.x;
      if (blk < p.nb && !*abort) p.drift[blk] = C.blocksum[2 * threadIdx.x] + C.blocksum[2 * threadIdx.x + 1];
    }
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kOCols);
  }
}

// A row-major bf16 matrix [rows, cols] as a 3-D tensor {cols, rows, 1}; box {64, box_rows, 1},
// 128-byte swizzle.  Loads past the edges read zeros; stores past them are dropped.
bool make_bf16_map(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int box_rows) {
  auto fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, 1};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)rows * cols * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count_of_device() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

template <int MODE>
cudaError_t launch_oproj_impl(const OProjArgs& a, cudaStream_t st) {
  const int K = a.H * 64;
  CUtensorMap ta, ta2, tb, tbp, tx, ty;
  if (!make_bf16_map(&ta, a.O, a.N, K, kOM) || !make_bf16_map(&tb, a.W_o, a.Dm, K, kON / 2))
    return cudaErrorInvalidValue;
  ta2 = ta;
  tx = ta;
  ty = ta;
  if (MODE == kDrift && !make_bf16_map(&ta2, a.O2, a.N, K, kOM)) return cudaErrorInvalidValue;
  if (MODE == kResidual) {
    if (!make_bf16_map(&ty, a.y, a.N, a.Dm, kOM)) return cudaErrorInvalidValue;
    if (a.x && !make_bf16_map(&tx, a.x, a.N, a.Dm, kOM)) return cudaErrorInvalidValue;
  }
  OParams p;
  p.N = a.N;
  p.K = K;
  p.Dm = a.Dm;
  p.nb = (a.N + 63) / 64;
  p.mtiles = (a.N + 2 * kOM - 1) / (2 * kOM);
  p.ntiles = (a.Dm + kON - 1) / kON;
  p.has_x = a.x != nullptr;
  p.drift = a.drift;
  p.status = a.status;
  const size_t smem = kOData + sizeof(OCtl) + 1024;
  cudaError_t e = cudaFuncSetAttribute(k_oproj<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int tiles = p.mtiles * p.ntiles, slots = max(1, sm_count_of_device() / 2);
  // Tiles past the last whole wave of pairs run as 2 or 4 units of fewer channels each where
  // those fit into one wave (43,968 tokens and d_model 1024: 688 tiles on 76 pairs are nine
  // waves and four tiles: 68.3 us with a tenth wave, 67.7 split, warm inputs).
  p.whole = tiles;
  p.parts = 1;
  const int left = tiles % slots;
  if (MODE == kResidual && left > 0 && 2 * left <= slots) {
    p.whole = tiles - left;
    p.parts = 4 * left <= slots ? 4 : 2;
  }
  const int units = p.whole + (tiles - p.whole) * p.parts;
  // Drift: one pair per stripe, persistent over the stripes, or a cluster of 2 or 4 pairs.  The
  // cost of a tile is its K / 64 steps and an epilogue of about two; starting and ending a CTA is
  // about eight, once for persistent pairs and for every wave of clusters.  A GPC rarely has room
  // for as many clusters of 8 CTAs as its SMs would allow, so those are counted with one in eight
  // less.  (16 heads, L2 flushed, persistent pairs / clusters of two / of four: 8 views 54.0 / 57.0 /
  // 49.9 us, 12 views 58.0 / 59.4 / 78.5, 16 views 103 / 84.6 / 95.9, 24 views 106 / 112 / 139, 32
  // views 152 / 138 / 183, 100 views 376 / 391 / 528.  84,608 tokens, 8 heads: 71.3 us with persistent
  // pairs, 83.9 with a pair launched per stripe.)
  p.group = 1;
  if (MODE == kDrift) {
    int64_t best = INT64_MAX;
    for (int g = 1; g <= 4 && g <= p.ntiles; g *= 2) {
      const int fit = max(1, g == 4 ? slots * 7 / 32 : slots / g);
      const int64_t waves = (p.mtiles + fit - 1) / fit, tile = p.K / 64 + 2;
      const int64_t run = (p.ntiles + g - 1) / g * tile;
      const int64_t cost = g == 1 ? waves * run + 8 : waves * (run + 8);
      if (cost < best) {
        best = cost;
        p.group = g;
      }
    }
  }
  const int ctas =
      2 * (p.group > 1 ? p.mtiles * p.group : min(MODE == kDrift ? p.mtiles : units, slots));
  tbp = tb;
  if (p.parts > 1 && !make_bf16_map(&tbp, a.W_o, a.Dm, K, kON / 2 / p.parts))
    return cudaErrorInvalidValue;
  return launch_with(k_oproj<MODE>, ctas, kOThreads, smem, st, true, 2 * p.group, ta, ta2, tb, tbp, tx,
                     ty, p);
}

}  // namespace

cudaError_t launch_out_proj(const OProjArgs& a, cudaStream_t st) {
  return launch_oproj_impl<kResidual>(a, st);
}

cudaError_t launch_token_drift(const OProjArgs& a, cudaStream_t st) {
  return launch_oproj_impl<kDrift>(a, st);
}

}  // namespace ress

// The row-by-block inner products of the selection on the tensor cores.  For one head and
// every candidate row i and block j, with x_i a per-row 64-vector and w_j a per-block one:
//   logits (Sec. 4.1):        L_ij = q_bar_i . k_bar_j / sqrt(64) * log2(e)  (j < nb)
//   drift norms (Eq. 9):      q_ij = ||y~_i||^2 + ||z~_j||^2 - 2 y~_i . z~_j   (j < nb)
//   round gains (Eq. 14/15):  t_ij = c_i - g~_i . z~_j,  c_i = y~_i . g~_i     (j < |P|)
// The rows P (as logits), q or t of the workspace receive the results.  The logits are kept
// in base-2 units, so that P_ij = 2^(L_ij - m_i) / Z_i; each 128-block slice of a row also
// yields its max and its sum of 2^(L - max), from which k_yagg assembles the softmax of the
// row (the pooled map P).
//
// Both operands are fp32; each is held as the sum of three bf16 terms (hi + mid + lo,
// written by the kernels that produce the vectors), and the product is accumulated in fp32
// TMEM from the six term products whose size is at least 2^-16 of hi.hi:
//   mid.mid + hi.lo + lo.hi + hi.mid + mid.hi + hi.hi      (smallest first)
// The three dropped products are below 2^-23 of |x||w| together, the size of the fp32
// rounding of the dot product itself.
//
// A tile is 128 rows x 128 blocks of one head.  k_dot, one CTA per tile, two per SM, 128 threads
// (logits) or 256:
//   thread 0   TMA of the six 128 x 64 bf16 term tiles (128-byte swizzle), two per mbarrier in
//              the order the products use them;
//   warp 0     converged MMA warp, one elected lane issues 6 x 4 tcgen05.mma M128 N128 K16
//              (A = x terms, B = w terms, both K-major from shared memory) and commits;
//   all warps  epilogue: tcgen05.ld of the accumulator rows (warp w: rows 32 (w mod 4)..), the
//              result into shared memory (the operand tiles are free by then) as boxes of 32
//              rows x 32 columns in the 128-byte-swizzled layout, each written out by its warp
//              with a TMA bulk tensor store as soon as it is formed (columns past the row
//              stride and rows past the array are clipped by the copy; rows past |P| are never
//              read).
// What bounds it is the chain of one tile (launch, loads, MMAs, epilogue, stores: about 6 us).
//
// k_dot_run, persistent CTAs, one per SM and 320 threads, each over a run of consecutive tiles
// (j fastest), so that the row terms stay in shared memory along a stripe of rows and the loads
// and products of a tile run under the epilogue of the one before:
//   warp 0     TMA: three block terms per tile (two stages), three row terms per stripe;
//   warp 1     the MMAs, into one of two accumulators;
//   warps 2-9  the epilogue, two boxes per warp on their way out, in two groups of four warps: a
//              half of each tile's columns each, or every other tile each where sums run along
//              the rows (logits).
// What bounds it is L2: 48 KB in and 64 KB out per tile, about 1.9 us (at 64 views a copy that
// stores every box twice takes 42 us instead of 28, one with a sixth of the MMAs 27).  Kernel times
// at 32 views (576 tiles): logits 14.7 -> 13.5 us, drift norms 14.9 -> 13.2, gains 14.9 -> 12.3
// against k_dot; at 100 views (4624 tiles) 98.8 -> 67.9, 94.5 -> 67.9 and 96 -> 64.6; all of a
// selection at 64 views (1936 tiles, six products) 1815 -> 1752 us.  Up to
// two tiles per SM k_dot is the better one: the layer at 8 views (64 tiles, 75% sparsity) takes 292
// us with it and 303 with k_dot_run, whose CTA needs more of the SM before it can start beside the
// kernel ahead of it; at 288 tiles (32 views, 128-token query blocks) they are equal, 1040 us.
// Every mbarrier wait is bounded; a wait that gives up records RESS_ETIMEOUT, lets copies and
// MMAs already issued finish (again bounded), frees TMEM and returns.

#include <cudaTypedefs.h>

#include "ress_internal.cuh"
#include "sm100_ptx.cuh"

namespace ress {
using namespace ptx;

namespace {

constexpr int kDotTile = 128;                     // rows i and blocks j per CTA
constexpr uint32_t kTermBytes = kDotTile * 128;   // 128 x 64 bf16
constexpr uint32_t kDotCols = 128;                // TMEM columns: one fp32 128 x 128 tile
constexpr uint32_t kRunCols = 256;                // two of them (runs of tiles)
constexpr uint32_t kBoxBytes = 32 * 32 * 4;       // 32 rows x 32 fp32 of the result
constexpr uint64_t kDotWaitNs = 2000000000ull;    // 2 s per wait
constexpr uint64_t kDotDrainNs = 200000000ull;    // 0.2 s to drain after an abort

enum DotMode { kDotGain = 0, kDotLogit = 1, kDotDist = 2 };
// One tile per CTA, epilogue warps: four, or eight (two per 32 rows, a half of the columns each)
// where no sum runs along the row.
template <int MODE>
constexpr int kDotThreads = MODE == kDotLogit ? 128 : 256;
constexpr int kRunWarps = 8;  // runs of tiles: epilogue warps
constexpr int kRunThreads = 64 + 32 * kRunWarps;
constexpr float kLogitScale = 0.125f * 1.4426950408889634f;  // 1/sqrt(64) * log2(e)

struct __align__(1024) DotSmem {
  uint8_t A[3][kTermBytes];  // row-vector terms (hi, mid, lo) of rows i0 .. i0 + 127
  uint8_t B[3][kTermBytes];  // block-vector terms of blocks j0 .. j0 + 127
  float bcol[kDotTile];      // drift norms: ||z~_j||^2 of the tile's blocks
  uint64_t full[3], done;  // operand terms by pairs, in the order the products need them
  uint32_t tmem_base;
  int abort;
};

struct __align__(1024) RunSmem {
  uint8_t A[3][kTermBytes];     // row-vector terms (hi, mid, lo) of the stripe's 128 rows
  uint8_t B[2][3][kTermBytes];  // block-vector terms of a tile's 128 blocks
  uint8_t box[kRunWarps][2][kBoxBytes];  // each epilogue warp's results on their way out
  float bcol[kRunWarps][kDotTile];       // drift norms: ||z~_j||^2 of the tile's blocks, per warp
  uint64_t full[2][3];  // operand terms by pairs, in the order the products need them
  uint64_t done[2];     // a tile's products are complete: accumulator full, operands free
  uint64_t free[2];     // the accumulator has been read
  uint32_t tmem_base;
  int abort;
};

struct DotParams {
  int nb;                // key blocks (columns)
  int nq, nqc;           // query blocks (rows), candidate query blocks
  int ni, nj, tiles;     // tiles of a head: ni x nj; of all heads
  const float* a;     // per row: c_i (gains) or ||y~_i||^2 (drift norms), [H, nb]
  const float* b;     // per block: ||z~_j||^2 (drift norms), [H, nb]
  float2* lstat;      // logits: per row and 128-block slice (max, sum 2^(L - max))
  int nslices;        // ceil(nb / 128)
  int ld;             // row stride of the output
  uint32_t* status;
  uint8_t head[RESS_MAX_HEADS];  // the heads with work, in order
};

struct DotTile {
  int h, i0, j0;
};

__device__ __forceinline__ DotTile dot_tile(const DotParams& p, int t) {
  const int s = t / p.nj;
  DotTile r;
  r.j0 = (t - s * p.nj) * kDotTile;
  r.h = p.head[s / p.ni];
  r.i0 = (s % p.ni) * kDotTile;
  return r;
}

// (A term, B term) of product q of the six, smallest first: 4 bits per q.
constexpr uint32_t kTermA = 0x010201u;  // q = 0..5 -> 1, 0, 2, 0, 1, 0
constexpr uint32_t kTermB = 0x001021u;  // q = 0..5 -> 1, 2, 0, 1, 0, 0

// Bounded wait by a whole warp (all lanes test once; otherwise lane 0 polls and broadcasts).
__device__ __forceinline__ bool dot_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                         uint64_t limit_ns) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort, limit_ns) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}

// 32 columns of a row of the result from the accumulator: o, and for the logits the running max
// and sum of 2^(L - max) over the row's slice.
template <int MODE>
__device__ __forceinline__ void dot_quarter(const uint32_t (&v)[32], float a, const float* bcol,
                                            int jq, int nb, float (&o)[32], float& pm, float& ps) {
  if (MODE == kDotGain) {
#pragma unroll
    for (int k = 0; k < 32; ++k) o[k] = a - __uint_as_float(v[k]);
  } else if (MODE == kDotLogit) {
    float cm = -INFINITY;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      o[k] = __uint_as_float(v[k]) * kLogitScale;
      if (jq + k < nb) cm = fmaxf(cm, o[k]);
    }
    if (cm > pm) {
      ps = (pm == -INFINITY) ? 0.f : ps * exp2f(pm - cm);
      pm = cm;
    }
    // the sum in four interleaved partial sums, with the SFU's exp2 (relative error
    // about 2^-22: far below what the row's softmax needs, and half the instructions)
    float sp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (jq + k < nb) sp[k & 3] += ex2(o[k] - pm);
    ps += (sp[0] + sp[1]) + (sp[2] + sp[3]);
  } else {
    // ||z~_j||^2 of the 32 blocks, broadcast from shared memory
    const float4* bq = reinterpret_cast<const float4*>(bcol);
#pragma unroll
    for (int k4 = 0; k4 < 8; ++k4) {
      const float4 bz = bq[k4];
      const float b4[4] = {bz.x, bz.y, bz.z, bz.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 4 * k4 + e;
        o[k] = fmaxf(fmaf(-2.0f, __uint_as_float(v[k]), a + b4[e]), 0.f);
      }
    }
  }
}

// Row `lane` of a box in the 128-byte-swizzled layout: 16-byte chunk k goes to k ^ (row mod 8).
__device__ __forceinline__ void box_row(uint8_t* box, int lane, const float (&o)[32]) {
  uint8_t* row = box + lane * 128;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    *reinterpret_cast<float4*>(row + ((k ^ (lane & 7)) << 4)) =
        make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
}

template <int MODE>
__global__ void __launch_bounds__(kDotThreads<MODE>)
    k_dot(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
          const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ DotParams p) {
  if (p.tiles == 0) {  // a round without swaps
    pdl_wait();
    return;
  }
  extern __shared__ uint8_t smem_raw[];
  DotSmem& S = *reinterpret_cast<DotSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                           ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &S.abort;
  const DotTile T = dot_tile(p, blockIdx.x);
  const int h = T.h, i0 = T.i0, j0 = T.j0;

  if (threadIdx.x == 0) {
    for (int t = 0; t < 3; ++t) mbar_init(&S.full[t], 1);
    mbar_init(&S.done, 1);
    S.abort = 0;
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
    prefetch_tensormap(&tmOut);
  }
  if (warp == 0) tmem_alloc(&S.tmem_base, kDotCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  if (MODE == kDotDist) {
    const int j = j0 + (int)threadIdx.x;
    if (threadIdx.x < kDotTile) S.bcol[threadIdx.x] = j < p.nb ? p.b[(int64_t)h * p.nb + j] : 0.f;
    __syncthreads();
  }
  const uint32_t tmem = S.tmem_base;

  bool issued = false;  // warp 0: MMAs went out (their completion must be awaited)
  if (warp == 0) {
    if (lane == 0) {
      // (mid, mid), (hi, lo), (lo, hi): the first products start while the others' terms land
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        const int ta = (kTermA >> (4 * t)) & 0xF, tb = (kTermB >> (4 * t)) & 0xF;
        mbar_arrive_expect_tx(&S.full[t], 2 * kTermBytes);
        tma_load_4d(S.A[ta], &tmA, &S.full[t], 0, i0, h, ta);
        tma_load_4d(S.B[tb], &tmB, &S.full[t], 0, j0, h, tb);
      }
    }
    __syncwarp();
    const bool leader = elect_one();
    if (__popc(__ballot_sync(0xffffffffu, leader)) != 1) {  // exactly one issuing lane
      if (lane == 0) {
        flag_status(p.status, kStatusBadRow);
        *abort = 1;
      }
    } else {
      const uint32_t idesc = idesc_bf16_f32(kDotTile, kDotTile, false);
      bool ok = true;
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        if (q < 3 && ok) {  // (the last three products use terms that have landed)
          ok = dot_wait(&S.full[q], 0, abort, kDotWaitNs);
          tc_fence_after();
        }
        if (ok && leader) {
          const uint32_t a = smem_u32(S.A[(kTermA >> (4 * q)) & 0xF]);
          const uint32_t b = smem_u32(S.B[(kTermB >> (4 * q)) & 0xF]);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_bf16_ss(tmem, sdesc_sw128(a + 32 * k), sdesc_sw128(b + 32 * k), idesc,
                        (q > 0 || k > 0) ? 1u : 0u);
          issued = true;
        }
        __syncwarp();
      }
      if (leader && issued) mma_commit(&S.done);
      issued = __any_sync(0xffffffffu, issued);
      if (!ok && lane == 0) {
        flag_status(p.status, kStatusTimeout);
        *abort = 1;
      }
    }
    if (*abort) {  // the copies must land before the shared memory goes away
      volatile int no_abort = 0;
      if (lane == 0)
        for (int t = 0; t < 3; ++t) mbar_wait(&S.full[t], 0, &no_abort, kDotDrainNs);
      __syncwarp();
    }
  }

  pdl_trigger();
  // ---- epilogue: warp w holds rows 32w .. 32w + 31 of the tile (TMEM lanes) ----------
  bool ok = dot_wait(&S.done, 0, abort, kDotWaitNs);
  if (!ok && lane == 0 && !*abort) {
    flag_status(p.status, kStatusTimeout);
    *abort = 1;
  }
  if (ok) {
    tc_fence_after();
    const int rw = warp & 3;            // this warp's 32 rows
    const int r = 32 * rw + lane;       // row of the tile = TMEM lane
    const int i = i0 + r;
    const int64_t ri = (int64_t)h * p.nq + i;
    float a = 0.f;
    if (MODE != kDotLogit && i < p.nq) a = p.a[ri];
    float pm = -INFINITY, ps = 0.f;  // logits: running max and sum over the slice
    uint8_t* stage = &S.A[0][0];     // 4 x 4 boxes of 32 rows x 32 fp32, 4 KB each
    constexpr int kQuarters = 512 / kDotThreads<MODE>;  // of 32 columns per warp
    const int q0 = kQuarters * (warp >> 2);
#pragma unroll 1
    for (int q = q0; q < q0 + kQuarters; ++q) {
      uint32_t v[32];
      __syncwarp();  // lane 0 comes from the store below
      RESS_TMEM_LD32(tmem + ((uint32_t)(32 * rw) << 16) + 32 * q, v);
      float o[32];
      dot_quarter<MODE>(v, a, S.bcol + 32 * q, j0 + 32 * q, p.nb, o, pm, ps);
      uint8_t* box = stage + q * 16384 + rw * 4096;
      box_row(box, lane, o);
      // this warp's box leaves while the next is formed
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && j0 + 32 * q < p.ld && i0 + 32 * rw < p.nq) {
        tma_store_3d(&tmOut, box, j0 + 32 * q, i0 + 32 * rw, h);
        bulk_commit();
      }
    }
    if (MODE == kDotLogit && i < p.nqc)
      p.lstat[ri * p.nslices + j0 / kDotTile] = make_float2(pm, ps);
    if (lane == 0) bulk_wait_read_all();  // the boxes are read before the shared memory goes away
    __syncwarp();
  }
  if (warp == 0 && issued && !ok) {  // MMAs still running: let them finish before the free
    volatile int no_abort = 0;
    if (lane == 0) mbar_wait(&S.done, 0, &no_abort, kDotDrainNs);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kDotCols);
  }
}

template <int MODE>
__global__ void __launch_bounds__(kRunThreads, 1)
    k_dot_run(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ DotParams p) {
  extern __shared__ uint8_t smem_raw[];
  RunSmem& S = *reinterpret_cast<RunSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                           ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort = &S.abort;
  // this CTA's tiles: t0 .. t0 + nt - 1
  const int t0 = (int)((int64_t)blockIdx.x * p.tiles / gridDim.x);
  const int nt = (int)((int64_t)(blockIdx.x + 1) * p.tiles / gridDim.x) - t0;
  constexpr int kGroups = MODE == kDotLogit ? 2 : 1;  // tiles in the epilogue at a time

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      for (int t = 0; t < 3; ++t) mbar_init(&S.full[s][t], 1);
      mbar_init(&S.done[s], 1);
      mbar_init(&S.free[s], kRunWarps / kGroups);
    }
    S.abort = 0;
    fence_barrier_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
    prefetch_tensormap(&tmOut);
  }
  if (warp == 1) tmem_alloc(&S.tmem_base, kRunCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  const uint32_t tmem = S.tmem_base;
  auto give_up = [&]() {
    if (!*abort) flag_status(p.status, kStatusTimeout);
    *abort = 1;
  };

  if (warp == 0) {
    // ---- producer: tile n's operands in stage n mod 2, free when tile n - 2 is done ------
    int n = 0;
    if (lane == 0) {
      bool ok = true;
      for (; n < nt && ok; ++n) {
        const int s = n & 1;
        if (n >= 2 && !mbar_wait(&S.done[s], ((n >> 1) - 1) & 1, abort, kDotWaitNs)) {
          give_up();
          break;
        }
        const DotTile T = dot_tile(p, t0 + n);
        const bool stripe = n == 0 || T.j0 == 0;  // new rows
#pragma unroll
        for (int t = 0; t < 3; ++t) {  // (mid, mid), (hi, lo), (lo, hi)
          const int ta = (kTermA >> (4 * t)) & 0xF, tb = (kTermB >> (4 * t)) & 0xF;
          mbar_arrive_expect_tx(&S.full[s][t], (stripe ? 2 : 1) * kTermBytes);
          if (n == 0) tma_load_4d(S.A[ta], &tmA, &S.full[s][t], 0, T.i0, T.h, ta);
          tma_load_4d(S.B[s][tb], &tmB, &S.full[s][t], 0, T.j0, T.h, tb);
        }
        if (stripe && n > 0) {  // the last stripe's products have read its row terms
          ok = mbar_wait(&S.done[s ^ 1], ((n - 1) >> 1) & 1, abort, kDotWaitNs);
          if (!ok) give_up();
#pragma unroll
          for (int t = 0; t < 3; ++t) {
            const int ta = (kTermA >> (4 * t)) & 0xF;
            if (ok) tma_load_4d(S.A[ta], &tmA, &S.full[s][t], 0, T.i0, T.h, ta);
          }
        }
      }
    }
    __syncwarp();
    pdl_trigger();
    if (lane == 0) {
      // copies in flight must land before the shared memory goes away: the MMA warp waits for
      // them as it goes, unless the CTA gave up
      if (nt > 0) mbar_wait(&S.done[(nt - 1) & 1], ((nt - 1) >> 1) & 1, abort, kDotWaitNs);
      if (*abort) {
        volatile int no_abort = 0;
        for (int m = n > 2 ? n - 2 : 0; m < n; ++m)
          for (int t = 0; t < 3; ++t)
            mbar_wait(&S.full[m & 1][t], (m >> 1) & 1, &no_abort, kDotDrainNs);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA: tile n into accumulator n mod 2 --------------------------------------------
    const bool leader = elect_one();
    int committed = 0;  // tiles whose products went out, at least in part
    if (__popc(__ballot_sync(0xffffffffu, leader)) != 1) {  // exactly one issuing lane
      if (lane == 0) {
        flag_status(p.status, kStatusBadRow);
        *abort = 1;
      }
    } else {
      const uint32_t idesc = idesc_bf16_f32(kDotTile, kDotTile, false);
      bool ok = true;
      for (int n = 0; n < nt && ok; ++n) {
        const int s = n & 1;
        if (n >= 2) ok = dot_wait(&S.free[s], ((n >> 1) - 1) & 1, abort, kDotWaitNs);
        tc_fence_after();
        bool issued = false;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          if (q < 3 && ok) {  // (the last three products use terms that have landed)
            ok = dot_wait(&S.full[s][q], (n >> 1) & 1, abort, kDotWaitNs);
            tc_fence_after();
          }
          if (ok && leader) {
            const uint32_t a = smem_u32(S.A[(kTermA >> (4 * q)) & 0xF]);
            const uint32_t b = smem_u32(S.B[s][(kTermB >> (4 * q)) & 0xF]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_bf16_ss(tmem + kDotTile * s, sdesc_sw128(a + 32 * k), sdesc_sw128(b + 32 * k),
                          idesc, (q > 0 || k > 0) ? 1u : 0u);
            issued = true;
          }
          __syncwarp();
        }
        if (leader && issued) mma_commit(&S.done[s]);
        if (__any_sync(0xffffffffu, issued)) committed = n + 1;
      }
      if (!ok && lane == 0) give_up();
    }
    pdl_trigger();
    if (committed > 0) {  // products still running finish before the accumulators are freed
      volatile int no_abort = 0;
      if (lane == 0)
        mbar_wait(&S.done[(committed - 1) & 1], ((committed - 1) >> 1) & 1, &no_abort,
                  *abort ? kDotDrainNs : kDotWaitNs);
      __syncwarp();
    }
  } else {
    // ---- epilogue: this warp's 32 rows are the TMEM lanes it can read --------------------
    const int ew = warp - 2, rw = warp & 3, group = ew >> 2;
    const int r = 32 * rw + lane;  // row of the tile = TMEM lane
    constexpr int kQuarters = MODE == kDotLogit ? 4 : 2;  // of 32 columns per warp and tile
    const int q0 = MODE == kDotLogit ? 0 : 2 * group;
    float* bcol = S.bcol[ew];
    bool ok = true;
    if ((MODE == kDotLogit ? group : 0) >= nt) pdl_trigger();
    for (int n = MODE == kDotLogit ? group : 0; n < nt && ok; n += kGroups) {
      const DotTile T = dot_tile(p, t0 + n);
      const int i = T.i0 + r;
      const int64_t ri = (int64_t)T.h * p.nq + i;
      float a = 0.f;
      if (MODE != kDotLogit && i < p.nq) a = p.a[ri];
      if (MODE == kDotDist) {
        __syncwarp();  // the last tile's norms have been read
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int k = 32 * (q0 + e) + lane, j = T.j0 + k;
          bcol[k] = j < p.nb ? p.b[(int64_t)T.h * p.nb + j] : 0.f;
        }
        __syncwarp();
      }
      if (n + kGroups >= nt) pdl_trigger();
      ok = dot_wait(&S.done[n & 1], (n >> 1) & 1, abort, kDotWaitNs);
      if (!ok) {
        if (lane == 0) give_up();
        break;
      }
      tc_fence_after();
      float pm = -INFINITY, ps = 0.f;  // logits: running max and sum over the slice
#pragma unroll 1
      for (int e = 0; e < kQuarters; ++e) {
        const int q = q0 + e;
        uint32_t v[32];
        __syncwarp();  // lane 0 comes from the store below
        RESS_TMEM_LD32(tmem + ((uint32_t)(32 * rw) << 16) + kDotTile * (n & 1) + 32 * q, v);
        if (e == kQuarters - 1) {  // read to the end: the accumulator is free
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&S.free[n & 1]);
        }
        float o[32];
        dot_quarter<MODE>(v, a, bcol + 32 * q, T.j0 + 32 * q, p.nb, o, pm, ps);
        uint8_t* box = S.box[ew][e & 1];
        if (lane == 0) bulk_wait_read_but1();  // this box's last copy has read it
        __syncwarp();
        box_row(box, lane, o);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (T.j0 + 32 * q < p.ld && T.i0 + 32 * rw < p.nq)
            tma_store_3d(&tmOut, box, T.j0 + 32 * q, T.i0 + 32 * rw, T.h);
          bulk_commit();  // (also where nothing left: groups are counted)
        }
      }
      if (MODE == kDotLogit && i < p.nqc)
        p.lstat[ri * p.nslices + T.j0 / kDotTile] = make_float2(pm, ps);
    }
    if (lane == 0) bulk_wait_read_all();  // the boxes are read before the shared memory goes away
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kRunCols);
  }
}

}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* q = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault,
                                         &r) == cudaSuccess &&
        r == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(q);
  }
  return fn;
}

// bf16 [3][H][nb][64] viewed as {64, nb, H, 3}; box {64, rows, 1, 1}, 128-byte swizzle.
// Rows past nb read as zeros.
bool make_term_map(CUtensorMap* m, const void* base, int nb, int H, int rows) {
  auto fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[4] = {64, (cuuint64_t)nb, (cuuint64_t)H, 3};
  cuuint64_t strides[3] = {128, (cuuint64_t)nb * 128, (cuuint64_t)H * nb * 128};
  cuuint32_t box[4] = {64, (cuuint32_t)rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 [H][nb][ld] viewed as {ld, nb, H}; box {32, rows, 1}, 128-byte swizzle.  Loads past
// the edges read zeros; stores past them are dropped.
bool make_row_map(CUtensorMap* m, void* base, int nb, int H, int ld, int rows) {
  auto fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)ld, (cuuint64_t)nb, (cuuint64_t)H};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 4, (cuuint64_t)nb * ld * 4};
  cuuint32_t box[3] = {32, (cuuint32_t)rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

template <int MODE>
cudaError_t launch_dot(const SelectArgs& a, int64_t a_terms, int64_t b_terms, int64_t out,
                       const float* rowv, const float* colv, int ncols, int round, float rho,
                       cudaStream_t st) {
  const Shape& s = a.s;
  if (s.ncand <= 0 || s.nqc <= 0) return cudaSuccess;
  CUtensorMap ta, tb, to;
  if (!make_term_map(&ta, a.ws + a_terms, s.nq, s.H, kDotTile) ||
      !make_term_map(&tb, a.ws + b_terms, s.nb, s.H, kDotTile) ||
      !make_row_map(&to, a.ws + out, s.nq, s.H, s.ld, 32))
    return cudaErrorInvalidValue;
  DotParams p;
  p.nb = s.nb;
  p.nq = s.nq;
  p.nqc = s.nqc;
  p.a = rowv;
  p.b = colv;
  p.lstat = (float2*)(a.ws + a.L.lstat);
  p.nslices = (s.nb + kDotTile - 1) / kDotTile;
  p.ld = s.ld;
  p.status = (uint32_t*)(a.ws + a.L.status);
  p.ni = (s.nqc + kDotTile - 1) / kDotTile;
  p.nj = (ncols + kDotTile - 1) / kDotTile;
  int heads = 0;  // a round swaps nothing in a head whose budget leaves no pair
  for (int h = 0; h < s.H; ++h)
    if (MODE != kDotGain || swap_count(a.c[h], s.ncand, round, rho) > 0)
      p.head[heads++] = (uint8_t)h;
  p.tiles = heads * p.ni * p.nj;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool run = p.tiles > 2 * sms;  // more than one wave of k_dot
  auto* kern = run ? k_dot_run<MODE> : k_dot<MODE>;
  const size_t smem = (run ? sizeof(RunSmem) : sizeof(DotSmem)) + 1024;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // (no tile: a round without swaps)
  const int ctas = run ? sms : p.tiles < 1 ? 1 : p.tiles;
  return launch_pdl(kern, ctas, run ? kRunThreads : kDotThreads<MODE>, smem, st, true, ta, tb, to,
                    p);
}

}  // namespace

cudaError_t launch_gain(const SelectArgs& a, int round, float rho, cudaStream_t st) {
  return launch_dot<kDotGain>(a, a.L.asplit, a.L.zsplit, a.L.t, (const float*)(a.ws + a.L.cdot),
                              nullptr, a.s.ncand, round, rho, st);
}

cudaError_t launch_logits(const SelectArgs& a, cudaStream_t st) {
  return launch_dot<kDotLogit>(a, a.L.asplit, a.L.ksplit, a.L.P, nullptr, nullptr, a.s.nb, 0,
                               0.f, st);
}

cudaError_t launch_drift_norms(const SelectArgs& a, cudaStream_t st) {
  return launch_dot<kDotDist>(a, a.L.asplit, a.L.zsplit, a.L.q, (const float*)(a.ws + a.L.ny),
                              (const float*)(a.ws + a.L.nz), a.s.nb, 0, 0.f, st);
}

}  // namespace ress

// Tensor-core projection GEMM of the attention path (bf16 operands, fp32
// accumulation) for sm_103a.
//
//   C[m, n] = sum_k A[m, k] B[n, k] + bias[n]        0 <= m < M, 0 <= n < N
//
// with A [rows, K] row-major (the block input for the query / key / value
// projection, the attention rows for the output projection) and B [N, K] a
// weight matrix.  Epilogues:
//   kProjQKV       N = 3D split into the attention's operand layouts: the q
//                  columns of token m go to row inv[m] of q_out (the token's
//                  place in the recomputing-token list; none if -1), the k
//                  columns to row m of k_out, and the v columns, transposed,
//                  to column m of vt_out [D, n_tok]
//   kProjResidual  row m belongs to token t = rows[m] (or m):
//                  a = bf16(C[m, :]), a_out[t, :] = a, u_out[t, :] = bf16(x[t, :] + a)
//                  (the attention output a_i and the MoE input u_i = x_i + a_i);
//                  u_i also goes to the token's FFN input rows when row_of is set
//   kProjResidualGated  as kProjResidual with u = bf16(x + g a), g the row's
//                  AdaLN gate (the sample's gate vector, Sec. 3); no FFN rows
// M is a host bound; when m_dev is set the launch reads the actual row count
// there (rows recomputed this step).
//
// Persistent CTA pairs (clusters of two, cta_group::2) as in the grouped FFN:
// a tile is 256 weight rows (the MMA's M side, 128 per CTA) by `n` token rows
// (its N side, half per CTA), two K sub-blocks of 64 per stage.  Tiles go to
// the pairs round robin, token tile by token tile.  11 warps per CTA:
//   warp 0    TMA producer of the weight boxes (128 rows);
//   warp 10   TMA producer of the token boxes (n / 2 rows);
//   warp 1    allocates 512 TMEM columns; in the leader, one thread issues
//             tcgen05.mma (M = 256, N = n, K = 16) for both CTAs into one of two
//             accumulators, so a tile's epilogue overlaps the next tile's MMAs;
//   warps 2-9 epilogue of the CTA's 128 features (TMEM lanes), two warps per
//             lane quadrant, each half of the token columns: 32 features x 32
//             tokens at a time through a 2 KB shared-memory stage, transposed
//             (except v^T, which wants the features' rows), so that each
//             global access covers 64 contiguous bytes of 8 rows.
// A kernel of single CTAs with one 128 x BN tile each was bound by its operand
// fill and by the CTAs' start and end.  Event-timed per launch on GB300, that
// one -> this one (4096 rows, cache steps with 60% of the rows listed):
//   D 1152 q/k/v 74 -> 32, 69 -> 28 us; output projection 49 -> 23, 42 -> 24 us
//   D 768 (2048 rows) q/k/v 19 -> 20, 16 -> 16 us; output 22 -> 14, 16 -> 15 us
// Every wait is bounded (about one second); a wait that runs out records the
// timeout status, raises a CTA abort flag, waits (bounded) for the copies and
// MMAs already issued, frees TMEM and returns.
#include <cuda.h>

#include <algorithm>
#include <new>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace moeca {

namespace {

constexpr int kBM = 128;                // weight rows per CTA (half of the MMA's M)
constexpr int kBK = 64;                 // K per sub-block
constexpr int kSub = 2;                 // K sub-blocks per stage
constexpr int kMaxN = 256;              // token rows per tile
constexpr int kBoxes = kMaxN / 32;      // token boxes of 16, 32, .., 128 rows
constexpr int kMaxStages = 5;
constexpr int kRingBytes = 208 * 1024;   // weight slots first, then token slots
constexpr int kEarly = 3;                // stages (every ring has as many) whose weights load before the wait
constexpr int kABytes = kBM * kBK * 2;  // 16 KB: one weight sub-block
constexpr int kWSlot = kSub * kABytes;  // a stage's weights
constexpr int kEpiWarps = 8;            // warps 2-9
constexpr int kTokWarp = 2 + kEpiWarps;
constexpr int kPThreads = 32 * (kTokWarp + 1);
constexpr int kStageOut = 32 * 64;      // per epilogue warp: 32 x 32 bf16
constexpr int kPSmem = kRingBytes + kEpiWarps * kStageOut + 1024;
constexpr int kTmemCols = 512;

struct ProjParams {
  int M, N, K;
  const int* m_dev;          // device row count (<= M), or null: M rows
  const float* bias;         // [N] or null
  const int32_t* rows;       // kProjResidual: token of row m, or null (m)
  int n_tok;                 // kProjResidual: tokens the x / a_out / u_out rows hold
  const __nv_bfloat16* x;    // kProjResidual: [n_tok, N]
  __nv_bfloat16* a_out;      // kProjResidual: [n_tok, N]
  __nv_bfloat16* u_out;      // kProjResidual: [n_tok, N]
  unsigned long long* row_stat;
  const int32_t* row_of;     // kProjResidual: [n_tok, row_w] FFN rows of the token (-1: none), or null
  int row_w;
  __nv_bfloat16* xg;         // [rows, N] FFN input rows that also take u
  const int32_t* inv;        // kProjQKV: list place of token m (-1: none), or null (m)
  __nv_bfloat16* q_out;      // kProjQKV: [list rows, D]
  __nv_bfloat16* k_out;      // kProjQKV: [n_tok, D]
  __nv_bfloat16* vt_out;     // kProjQKV: [D, n_tok]
  const float* gate;         // kProjResidualGated: gate row of token t at gate + (t / seq) * gate_ld
  int gate_ld, seq;
  int first;                 // 1: no weights before the dependency wait (see ProjArgs)
  int* status;
};

struct ProjMaps {
  CUtensorMap w;             // weights, box 128 rows
  CUtensorMap act[kBoxes];   // token rows, boxes of 16 .. 128 rows
};

// Token tile width for `rows` rows: the fewest waves x time per tile.  A
// tile's time per stage is modelled as 384 + n: the MMAs alone take n / 2
// clocks each (64 at 128 columns, 128 at 256, at least 45), but the
// single-thread roles' work per stage and the barrier round trips do not
// depend on n, so that narrow tiles save less than their share.
__host__ __device__ __forceinline__ int token_width(int rows, int nw, int pairs) {
  int best = 256, best_cost = 0x7fffffff;
  for (int n = 256; n >= 32; n -= 32) {
    const int tiles = (rows + n - 1) / n * nw;
    const int cost = (tiles + pairs - 1) / pairs * (384 + n);
    if (cost < best_cost) {
      best_cost = cost;
      best = n;
    }
  }
  return best;
}

// A warp's 32 features (lanes) x 32 tokens as bf16 into the stage as
// [32 features][32 tokens], 16-byte chunks XOR-swizzled by row
// pairs so that both accesses are conflict-free.
__device__ __forceinline__ void stage_by_feature(uint32_t* stage, const uint32_t* v, float bias, int lane) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint4 w;
    uint32_t* wp = reinterpret_cast<uint32_t*>(&w);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      wp[q] = pack_bf16(__uint_as_float(v[8 * j + 2 * q]) + bias, __uint_as_float(v[8 * j + 2 * q + 1]) + bias);
    reinterpret_cast<uint4*>(stage)[lane * 4 + (j ^ ((lane >> 1) & 3))] = w;
  }
}

template <int MODE>
__global__ void __launch_bounds__(kPThreads, 1)
    proj_tc_kernel(const __grid_constant__ ProjMaps maps, const ProjParams p) {
  constexpr bool kRes = MODE != kProjQKV;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];  // leader's: the stage's bytes of both CTAs
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t tfull_bar[2];
  __shared__ __align__(8) uint64_t tempty_bar[2];         // leader's: the epilogue warps of both CTAs
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_sh;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&tfull_bar[s]), 1);
      mbar_init(smem_u32(&tempty_bar[s]), 2 * kEpiWarps);
    }
    mbar_init(smem_u32(&drain_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  if (warp == 2 && lane <= kBoxes) {
    const CUtensorMap* t = lane ? &maps.act[lane - 1] : &maps.w;
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(t)) : "memory");
  }
  cluster_arrive();
  cluster_wait();  // both CTAs' barriers are initialised, TMEM is allocated
  tc_fence_after();
  const uint32_t ring = smem_u32(smem);
  const int nw = (p.N + 2 * kBM - 1) / (2 * kBM);
  const int sub = p.K / kBK, ks = (sub + kSub - 1) / kSub;
  // The weights of the first tile's first stages load before the dependency
  // wait: which they are does not depend on the row count.  Their bytes
  // complete on the stages' barriers, which the leader arms after the wait.
  // Not in a step's first launch: a caller's kernel right before it that wrote
  // the weights has ended then, but only the wait makes its writes visible.
  const int early = p.first ? 0 : min(kEarly, ks), w_first = pair % nw;
  if (warp == 0 && lane == 0) {
    const int feat = w_first * 2 * kBM + static_cast<int>(rank) * kBM;
    const uint32_t full0 = cluster_addr(smem_u32(&full_bar[0]), 0);
    for (int k = 0; k < early; ++k)
      tma_load_k64_pair(ring + k * kWSlot, &maps.w, feat, k * kSub, full0 + k * 8);
  }
  pdl_entry();
  const int M = p.m_dev ? min(*reinterpret_cast<const volatile int*>(p.m_dev), p.M) : p.M;
  if (p.row_stat && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(p.row_stat, static_cast<unsigned long long>(M));
  const uint32_t tmem = tmem_sh;
  const int n = token_width(M, nw, n_pairs), half = n >> 1;
  const int units = (M + n - 1) / n * nw;
  const int t_slot = kSub * half * (kBK * 2);  // a stage's token rows
  const int nst = min(kMaxStages, kRingBytes / (kWSlot + t_slot));
  const uint32_t ring_t = ring + nst * kWSlot;
  const uint32_t empty0 = smem_u32(&empty_bar[0]);

  if (warp == 0 || warp == kTokWarp) {
    if (lane == 0) {
      // ---------------- TMA producers: weights (warp 0), tokens ----------------
      const bool wts = warp == 0;
      const CUtensorMap* map = wts ? &maps.w : &maps.act[(n >> 5) - 1];
      const int slot_bytes = wts ? kWSlot : t_slot;
      const uint32_t first = wts ? ring : ring_t, end = first + nst * slot_bytes;
      const uint32_t full0 = cluster_addr(smem_u32(&full_bar[0]), 0);
      uint32_t dst = first, eb = empty0, fb = full0, par = 1u;
      int issued = 0;
      bool ok = true;
      for (int u = pair; u < units && ok; u += n_pairs) {
        const int tt = u / nw, w = u - tt * nw;
        const int feat = w * 2 * kBM + static_cast<int>(rank) * kBM;
        const int row = wts ? feat : tt * n + static_cast<int>(rank) * half;
        // Bytes a stage brings into both CTAs (rows and sub-blocks past the last
        // are zero-filled).  A half tile without weight rows is copied as well: a
        // CTA that brought nothing could be lapped by the MMAs, and a barrier two
        // phases on looks like one not yet completed.
        const uint32_t tx = 2 * kWSlot + kSub * n * (kBK * 2);
        for (int k = 0; k < ks; ++k) {
          // The slot is free in both CTAs once the MMAs that read it are done;
          // the leader arms its barrier with the bytes of both CTAs.
          if (!(ok = mbar_wait_hot(eb, par, &abort_flag))) break;
          if (wts && rank == 0) mbar_expect_tx(fb, tx);
          if (!(wts && issued < early)) tma_load_k64_pair(dst, map, row, k * kSub, fb);
          ++issued;
          dst += slot_bytes;
          eb += 8;
          fb += 8;
          if (dst == end) {
            dst = first;
            eb = empty0;
            fb = full0;
            par ^= 1u;
          }
        }
      }
      if (wts && rank == 0 && pair >= units) {
        // No tile for this pair: the early copies land before the CTAs exit.
        for (int k = 0; k < early; ++k) mbar_expect_tx(smem_u32(&full_bar[k]), 2 * kWSlot);
        for (int k = 0; k < early && ok; ++k) ok = mbar_wait(smem_u32(&full_bar[k]), 0, &abort_flag);
      }
      if (!ok) {
        if (!abort_flag) report_status(p.status, kStatusWaitTimeout, wts ? 600 : 603);
        abort_flag = 1;
        // Copies already issued land before the CTAs can exit: the newest use
        // of every slot (the leader's barriers see both CTAs').
        for (int q = 0; wts && rank == 0 && q < nst && q < issued; ++q) {
          const int last = issued - 1 - (issued - 1 - q) % nst;
          const unsigned long long t0 = globaltimer();
          while (!mbar_try(smem_u32(&full_bar[q]), (last / nst) & 1) && globaltimer() - t0 < kTcWaitNs) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // ---------------- MMA issuer (the leader, for both CTAs) ----------------
      const uint32_t w_lo0 = ((ring & 0x3FFFFu) >> 4) | (1u << 16), x_lo0 = ((ring_t & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t full0 = smem_u32(&full_bar[0]);
      const uint32_t idesc = instr_desc(2 * kBM, n), b_sub = n * kBK >> 4;
      const uint32_t x_end = x_lo0 + nst * (static_cast<uint32_t>(t_slot) >> 4);
      uint32_t w_lo = w_lo0, x_lo = x_lo0, fb = full0, eb = empty0, par = 0u, acc_phase = 0;
      int acc = 0;
      bool ok = true;
      for (int u = pair; u < units; u += n_pairs) {
        if (!(ok = mbar_wait(smem_u32(&tempty_bar[acc]), acc_phase ^ 1u, &abort_flag))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + static_cast<uint32_t>(acc * kMaxN);
        for (int k = 0; k < ks; ++k) {
          if (!(ok = mbar_wait_hot(fb, par, &abort_flag))) break;
          tc_fence_after();
#pragma unroll
          for (int q = 0; q < kSub; ++q) {
            if (q && k * kSub + q >= sub) break;
            const uint32_t wq = w_lo + q * (kABytes >> 4), xq = x_lo + q * b_sub;
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              mma_bf16_pair(d_tmem, wq + kk * 2, xq + kk * 2, idesc, k != 0 || q != 0 || kk != 0);
          }
          mma_commit_pair(eb);
          w_lo += kWSlot >> 4;
          x_lo += static_cast<uint32_t>(t_slot) >> 4;
          fb += 8;
          eb += 8;
          if (x_lo == x_end) {
            w_lo = w_lo0;
            x_lo = x_lo0;
            fb = full0;
            eb = empty0;
            par ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit_pair(smem_u32(&tfull_bar[acc]));
        if (++acc == 2) {
          acc = 0;
          acc_phase ^= 1u;
        }
      }
      if (!ok) {
        if (!abort_flag) report_status(p.status, kStatusWaitTimeout, 601);
        abort_flag = 1;
      }
      // Every MMA issued so far has completed once the drain barrier fires.
      mma_commit_pair(smem_u32(&drain_bar), 1);
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(smem_u32(&drain_bar), 0) && globaltimer() - t0 < kTcWaitNs) {
      }
    }
  } else {
    // ---------------- Epilogue ----------------
    const int quad = warp & 3;           // TMEM lanes [32 quad, 32 quad + 32)
    const int part = (warp - 2) >> 2;    // which half of the tile's token columns
    uint32_t* stage = reinterpret_cast<uint32_t*>(smem + kRingBytes + (warp - 2) * kStageOut);
    const uint32_t tempty0 = cluster_addr(smem_u32(&tempty_bar[0]), 0);
    const int s_row = lane >> 2, s_ch = lane & 3;  // this lane's row (of 8) and 16-byte chunk of a staged store
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int u = pair; u < units; u += n_pairs) {
      const int tt = u / nw, w = u - tt * nw;
      const int feat = w * 2 * kBM + static_cast<int>(rank) * kBM + quad * 32;  // the warp's 32 features
      const int m0 = tt * n;
      const int c_lo = part * half, c_hi = feat < p.N ? min(c_lo + half, M - m0) : 0;
      const float bias = p.bias && feat < p.N ? __ldg(p.bias + feat + lane) : 0.f;
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&tfull_bar[acc]), acc_phase, &abort_flag)))) break;
      tc_fence_after();
      const uint32_t tb = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(acc * kMaxN);
#pragma unroll 1
      for (int c = c_lo; c < c_hi; c += 32) {
        // This lane's token of the chunk (c + lane) and the row its values go to.
        const int m = m0 + c + lane;
        int row = -1;
        if (c + lane < c_hi) {
          if constexpr (kRes) {
            row = p.rows ? p.rows[m] : m;
            if (row < 0 || row >= p.n_tok) {
              report_status(p.status, kStatusBadIndex, 6000000 + m);
              row = -1;
            }
          } else {
            row = m;
          }
        }
        uint32_t v[32];
        tmem_ld32_async(tb + c, v);
        if constexpr (kRes) {
          // The residual input rows in the staged stores' layout, in flight
          // while the tile is read and staged.
          uint4 xv[4];
          int tok[4];
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            tok[it] = __shfl_sync(0xffffffffu, row, it * 8 + s_row);
            if (tok[it] >= 0)
              xv[it] = __ldg(reinterpret_cast<const uint4*>(p.x + static_cast<size_t>(tok[it]) * p.N + feat + s_ch * 8));
          }
          tmem_wait32(v);
          __syncwarp();
          stage_by_token(stage, lane, [&](int t) { return __uint_as_float(v[t]) + bias; });
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            const uint4 av = *reinterpret_cast<const uint4*>(stage + (it * 8 + s_row) * 16 + s_ch * 4);
            if (tok[it] < 0) continue;
            const size_t off = static_cast<size_t>(tok[it]) * p.N + feat + s_ch * 8;
            float gg[8];
            if constexpr (MODE == kProjResidualGated) {
              const float* g = p.gate + static_cast<size_t>(tok[it] / p.seq) * p.gate_ld + feat + s_ch * 8;
              const float4 g0 = __ldg(reinterpret_cast<const float4*>(g));
              const float4 g1 = __ldg(reinterpret_cast<const float4*>(g) + 1);
              gg[0] = g0.x; gg[1] = g0.y; gg[2] = g0.z; gg[3] = g0.w;
              gg[4] = g1.x; gg[5] = g1.y; gg[6] = g1.z; gg[7] = g1.w;
            }
            uint4 uv;
            const __nv_bfloat162* ah = reinterpret_cast<const __nv_bfloat162*>(&av);
            const __nv_bfloat162* xh = reinterpret_cast<const __nv_bfloat162*>(&xv[it]);
            __nv_bfloat162* uh = reinterpret_cast<__nv_bfloat162*>(&uv);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float2 af = __bfloat1622float2(ah[q]), xf = __bfloat1622float2(xh[q]);
              if constexpr (MODE == kProjResidualGated)
                uh[q] = __floats2bfloat162_rn(fmaf(gg[2 * q], af.x, xf.x), fmaf(gg[2 * q + 1], af.y, xf.y));
              else
                uh[q] = __floats2bfloat162_rn(xf.x + af.x, xf.y + af.y);
            }
            *reinterpret_cast<uint4*>(p.a_out + off) = av;
            *reinterpret_cast<uint4*>(p.u_out + off) = uv;
            if constexpr (MODE == kProjResidual) {
              const int n_g = p.row_of ? p.row_w : 0;
              for (int q = 0; q < n_g; ++q) {
                const int pos = __ldg(p.row_of + static_cast<size_t>(tok[it]) * p.row_w + q);
                if (pos >= 0) *reinterpret_cast<uint4*>(p.xg + static_cast<size_t>(pos) * p.N + feat + s_ch * 8) = uv;
              }
            }
          }
        } else {
          // The warp's features lie in one of q, k, v (D is a multiple of 64).
          const int Dm = p.N / 3, region = feat / Dm, f = feat - region * Dm;
          if (region == 0 && row >= 0 && p.inv) row = p.inv[m];
          tmem_wait32(v);
          __syncwarp();
          if (region < 2) {
            stage_by_token(stage, lane, [&](int t) { return __uint_as_float(v[t]) + bias; });
            __syncwarp();
            __nv_bfloat16* base = (region == 0 ? p.q_out : p.k_out) + f + s_ch * 8;
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const uint4 val = *reinterpret_cast<const uint4*>(stage + (it * 8 + s_row) * 16 + s_ch * 4);
              const int r = __shfl_sync(0xffffffffu, row, it * 8 + s_row);
              if (r >= 0) *reinterpret_cast<uint4*>(base + static_cast<size_t>(r) * Dm) = val;
            }
          } else {
            // v^T: rows are features; 8 consecutive tokens per lane (the token
            // count is a multiple of 8).
            stage_by_feature(stage, v, bias, lane);
            __syncwarp();
            __nv_bfloat16* base = p.vt_out + static_cast<size_t>(f) * p.n_tok + m0 + c + s_ch * 8;
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const int fr = it * 8 + s_row;
              const uint4 val = reinterpret_cast<const uint4*>(stage)[fr * 4 + (s_ch ^ ((fr >> 1) & 3))];
              if (c + s_ch * 8 < c_hi) *reinterpret_cast<uint4*>(base + static_cast<size_t>(fr) * p.n_tok) = val;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty0 + acc * 8);
      if (++acc == 2) {
        acc = 0;
        acc_phase ^= 1u;
      }
    }
    if (!ok) {
      if (lane == 0 && !abort_flag) report_status(p.status, kStatusWaitTimeout, 602);
      abort_flag = 1;
    }
  }
  // Neither CTA leaves (or frees TMEM) while the other may still reach its
  // shared memory or the pair's MMAs run.
  tc_fence_before();
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

struct ProjPlan {
  ProjMaps maps;
  int N, K;
  bool rows;  // the token maps are set
};

ProjPlan* proj_plan_create(const void* w, int N, int K, const void* A, int a_rows) {
  if (N % 64 || K % 64) return nullptr;
  ProjPlan* p = new (std::nothrow) ProjPlan{};
  if (!p) return nullptr;
  p->N = N;
  p->K = K;
  p->rows = A != nullptr;
  bool ok = encode_k64(&p->maps.w, w, static_cast<uint64_t>(N), static_cast<uint64_t>(K), kBM, kSub);
  for (int i = 0; i < kBoxes && ok && A; ++i)
    ok = encode_k64(&p->maps.act[i], A, static_cast<uint64_t>(a_rows), static_cast<uint64_t>(K), 16 * (i + 1), kSub);
  if (ok) return p;
  delete p;
  return nullptr;
}

void proj_plan_destroy(ProjPlan* p) { delete p; }

cudaError_t launch_proj_tc(const ProjPlan* plan, const ProjArgs& a, int n_sms, cudaStream_t s) {
  if (!plan || a.M <= 0 || (!a.A && !plan->rows)) return cudaErrorInvalidValue;
  if (a.mode == kProjResidualGated && (!a.gate || a.seq <= 0 || a.row_of)) return cudaErrorInvalidValue;
  const int N = plan->N, K = plan->K;
  // At most one pair per tile of the narrowest width.
  const int nw = (N + 2 * kBM - 1) / (2 * kBM);
  const int pairs = std::max(1, std::min(n_sms / 2, (a.M + 31) / 32 * nw));
  ProjMaps maps = plan->maps;
  if (a.A) {
    // The caller's rows (a step's input): the one width the launch will take
    // when the host knows the row count, else all of them.
    const int only = a.m_dev ? 0 : token_width(a.M, nw, pairs) / 32;
    for (int i = 0; i < kBoxes; ++i) {
      if (only && i) {
        maps.act[i] = maps.act[0];
      } else if (!encode_k64(&maps.act[i], a.A, static_cast<uint64_t>(a.a_rows), static_cast<uint64_t>(K),
                             16 * (only ? only : i + 1), kSub)) {
        return cudaErrorInvalidValue;
      }
    }
  }
  ProjParams p{};
  p.M = a.M; p.N = N; p.K = K; p.m_dev = a.m_dev; p.bias = a.bias;
  p.rows = a.rows; p.n_tok = a.n_tok;
  p.x = static_cast<const __nv_bfloat16*>(a.x);
  p.a_out = static_cast<__nv_bfloat16*>(a.a_out);
  p.u_out = static_cast<__nv_bfloat16*>(a.u_out);
  p.row_stat = a.row_stat;
  p.row_of = a.row_of;
  p.row_w = a.row_w;
  p.xg = static_cast<__nv_bfloat16*>(a.xg);
  p.inv = a.inv;
  p.q_out = static_cast<__nv_bfloat16*>(a.q_out);
  p.k_out = static_cast<__nv_bfloat16*>(a.k_out);
  p.vt_out = static_cast<__nv_bfloat16*>(a.vt_out);
  p.gate = a.gate; p.gate_ld = a.gate_ld; p.seq = a.seq;
  p.first = a.first;
  p.status = a.status;
  auto run = [&](auto kern) -> cudaError_t {
    const cudaError_t e = set_dyn_smem_on_device(reinterpret_cast<const void*>(kern), kPSmem);
    if (e != cudaSuccess) return e;
    return launch_pdl<2>(kern, dim3(2 * pairs), dim3(kPThreads), kPSmem, s, maps, p);
  };
  switch (a.mode) {
    case kProjQKV: return run(proj_tc_kernel<kProjQKV>);
    case kProjResidual: return run(proj_tc_kernel<kProjResidual>);
    case kProjResidualGated: return run(proj_tc_kernel<kProjResidualGated>);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace moeca

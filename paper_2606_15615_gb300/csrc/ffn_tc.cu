// Tensor-core grouped expert FFN (bf16 operands, fp32 accumulation) for sm_103a.
//
// Computes the recompute branches of Eq. 5 / Eq. 6 over the compacted rows:
//   phase 1: hmid[r, :] = GELU(xg[r, :] W1_g^T)         N = F, K = D
//   phase 2: dst[list[r], :] = hmid[r, :] W2_g^T         N = D, K = F
// where rows r of expert group g are [offsets[g], offsets[g] + counts[g]) and
// dst is the branch cache (token*k + slot) or the shared-expert rows.
//
// Persistent kernel on CTA pairs (clusters of two, cta_group::2), one CTA per
// SM.  A tile is 256 weight rows by up to 256 token rows: the weights are the
// MMA's M side (128 rows per CTA), the token rows its N side (each CTA holds
// half), so a group's token tile is as wide as its rows need (rounded up to
// 32) and its weights are read once per 256 token rows.  What bounds the
// kernel at many rows is how fast an SM fills its operands (and the
// shared-memory bandwidth that the copies and the MMAs share): per 128 weight
// rows of output and 64 of K a CTA brings in 128 + n / 2 rows of 128 bytes,
// where single CTAs with token rows on M brought in 128 + 128 x 128 / BN
// per token tile of 128.  With few rows per expert the weight stream binds:
// about 5.5 TB/s while tiles run, with gaps at the start and between the two
// GEMMs.  Event-timed per launch on GB300, single-CTA kernel -> this one,
// full step / cache step at ~60% reuse:
//   D 2560, 4 + 1 experts, F 6912, T 4096   627 -> 510 / 370 -> 300 us
//   D 1152, 16 experts, F 4608, T 4096      188 -> 155 / 101 ->  92 us
//   D 1152, 64 experts top-8, F 768, T 4096 163 -> 125 /  86 ->  66 us
//   D 1024, 32 experts top-4, F 1600, T 1157 92 ->  56 /  62 ->  49 us
//   D 768, 16 experts, F 3072, T 2048        61 ->  61 /  45 ->  44 us
// (870 GFLOP in 510 us at D 2560: 0.89 of the measured bf16 rate.)
// 12 warps per CTA:
//   warp 0  TMA producer of the CTA's weight boxes (128 rows x 64, 128-byte
//           swizzle, two K sub-blocks per copy), completing on the leader's
//           barriers; the leader's also hands out the units.  The weights
//           depend on no other unit, so in phase 2 they run ahead while the
//           hidden rows are still being written;
//   warp 10 TMA producer of the token boxes (n / 2 rows); in phase 2 it waits
//           for the tile's hidden rows;
//   warp 1  allocates 512 TMEM columns; in the leader, one thread issues
//           tcgen05.mma (M = 256, N = n, K = 16) for both CTAs;
//           tcgen05.commit frees the stage in both and signals a finished
//           accumulator;
//   warps 2-9  epilogue of the CTA's 128 weight rows (TMEM lanes), two warps
//           per lane quadrant, each half of the token columns: tcgen05.ld,
//           GELU / bf16 rounding, a transpose through shared memory, row
//           stores (phase 2 scatters through the row list);
//   warp 11 publishes stored phase-1 tiles to phase 2 (a GPU-scope release
//           takes about a microsecond, which the epilogue need not wait for).
// The single-thread roles run their loops at some five cycles an instruction,
// so a stage's instructions count: running addresses, one copy per operand
// and stage (K in 3-D sub-blocks), the first try of a wait inline, units
// decoded once (by the leader's weight producer) and passed on whole.  Code
// size counts as well: each launch fetches its code anew, and while the first
// weights stream in a fetch is slow (a second, unrolled copy of the epilogue
// cost 2% of a D 768 step, functions called out of line 5%).  Tried and not
// better: 64 of K per stage, 16 epilogue warps, L2 prefetches of the weights
// 4 or 8 stages ahead (1-4% slower each).
// Two TMEM accumulators (2 x 256 columns) let the epilogue of one tile
// overlap the MMAs of the next.  Units run token tile by token tile, weight
// tiles minor.  Group sizes stay on the device: every CTA derives the tile
// list from them.
//
// Every mbarrier wait is bounded (about one second of %globaltimer); a wait
// that runs out records MOECA's timeout status, raises a CTA-wide abort flag,
// drains the copies and MMAs this CTA issued, frees TMEM and returns.
#include <cuda.h>
#include <algorithm>
#include <cstdio>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace moeca {

namespace {

constexpr int kBM = 128;          // weight rows per CTA (half of the MMA's M)
constexpr int kBK = 64;           // K per sub-block: 64 bf16 = one 128-byte swizzle row
constexpr int kSub = 2;           // K sub-blocks per stage
constexpr int kMaxN = 256;        // token rows per tile
constexpr int kMaxStages = 5;     // what the ring holds at the narrowest token tile (32 rows)
constexpr int kRingBytes = 208 * 1024;  // beside 16 KB of epilogue stages
constexpr int kEpiWarps = 8;        // warps 2-9
constexpr int kTokWarp = 2 + kEpiWarps;
constexpr int kPubWarp = kTokWarp + 1;
constexpr int kThreads = 32 * (kPubWarp + 1);
constexpr int kTmemCols = 512;
constexpr int kABytes = kBM * kBK * 2;  // 16 KB: one weight sub-block
constexpr int kStageOut = 32 * 64;      // per epilogue warp: 32 tokens x 32 features of bf16
constexpr int kSmemBytes = kRingBytes + kEpiWarps * kStageOut + 1024;
static_assert(kMaxStages == kRingBytes / (kSub * (kABytes + 32 / 2 * (kBK * 2))), "stages at the narrowest tile");
constexpr int kMaxGroups = kMaxExperts + 1;
constexpr unsigned long long kWaitNs = 1000000000ull;
constexpr int kUQ = 4;            // unit queue from the leader's producer to the other roles
constexpr int kBoxes = kMaxN / 32;  // token boxes of 16, 32, .., 128 rows

struct TcArgs {
  int G, E, k, T;
  int N[2];          // per phase: output width
  int K[2];          // per phase: contraction length
  int cap;           // widest token tile (a multiple of 32, at most 256)
  int split;         // K splits of phase 2
  int units_max;     // split-K units the workspace holds
  const int32_t* counts;
  const int32_t* offsets;
  const int32_t* list;
  void* hmid;      // phase 1 output [rows, F]
  void* cache_h;   // phase 2 routed destination [T*k, D]
  void* shared_h;  // phase 2 shared destination [T, D]
  float* partial;  // split-K partial tiles, one [256][128] fp32 slice per CTA and unit
  int* tile_sem;   // split-K arrival counters, one per epilogue warp of a half tile, left at 0
  int* dep;        // per token tile {phase-1 half tiles stored, phase-2 CTAs started}, left at 0
  int dep_pairs;   // capacity of dep (pairs)
  int* work;       // next unit ticket; the kernel after this one re-arms it to 0 (launch_ffn_tc's contract)
  int* status;
};

// Tensor maps of one phase: routed and shared weights (box 128 rows) and the
// token rows in boxes of 16 .. 128 rows (half a tile of 32 .. 256).
struct TcMaps {
  CUtensorMap w, ws;
  CUtensorMap act[kBoxes];
};
struct TcMapPair {
  TcMaps p[2];
};

// Tanh-form GELU with the hardware tanh approximation (MUFU; relative error
// about 2^-11).  The result is rounded to bf16 (relative step 2^-8) right
// after, so the approximation stays below the output rounding.
__device__ __forceinline__ float gelu_tanh_hw(float z) {
  const float u = 0.7978845608028654f * fmaf(0.044715f * z, z * z, z);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  const float hz = 0.5f * z;
  return fmaf(hz, t, hz);
}

// A phase's geometry for this launch.
struct Phase {
  int nw;   // weight tiles of 256 rows (the last may be short)
  int ks;   // stages (K / (64 kSub), rounded up)
  int sub;  // K sub-blocks
  int S;    // K splits
  int units;
};

// One unit of work: phase p, group g, weight tile w, token tile tt (index over
// all groups) of n columns, `valid` of them rows, from row row0 on; K split sp.
struct Unit {
  int p, sp, g, n, valid, tt, w, row0;
};

// A unit as the queue carries it; x is negative after the last unit.
__device__ __forceinline__ int4 pack_unit(const Unit& t) {
  return make_int4(t.p | (t.sp << 1) | (t.g << 4) | ((t.n >> 5) << 12) | ((t.valid - 1) << 16), t.tt, t.w, t.row0);
}
__device__ __forceinline__ Unit unpack_unit(const int4& v) {
  Unit t;
  t.p = v.x & 1;
  t.sp = (v.x >> 1) & 7;
  t.g = (v.x >> 4) & 127;
  t.n = ((v.x >> 12) & 15) << 5;
  t.valid = ((v.x >> 16) & 255) + 1;
  t.tt = v.y;
  t.w = v.z;
  t.row0 = v.w;
  return t;
}

// Group tables of the launch, in shared memory.
struct Groups {
  int before[kMaxGroups + 1];  // token tiles ahead of each group; [G] = all
  int cnt[kMaxGroups];
  int off[kMaxGroups];
  int wid[kMaxGroups];         // token tile width
};

__device__ __forceinline__ Unit decode_unit(int u, const Phase& p0, const Phase& p1, const Groups& gr, int G) {
  Unit r;
  r.p = u < p0.units ? 0 : 1;
  int v = u - (r.p ? p0.units : 0);
  const int nw = r.p ? p1.nw : p0.nw, S = r.p ? p1.S : p0.S;
  r.sp = 0;
  if (S > 1) {
    const int t = v / S;
    r.sp = v - t * S;
    v = t;
  }
  r.tt = v / nw;
  r.w = v - r.tt * nw;
  // Last group whose first token tile is at or before tt (empty groups
  // precede the non-empty group that shares their start).
  int lo = 0, hi = G - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (gr.before[mid] <= r.tt) lo = mid;
    else hi = mid - 1;
  }
  r.g = lo;
  r.n = gr.wid[lo];
  const int first = (r.tt - gr.before[lo]) * r.n;
  r.valid = min(r.n, gr.cnt[lo] - first);
  r.row0 = gr.off[lo] + first;
  return r;
}

// The queue's word of unit u (negative past the last).
__device__ __forceinline__ int4 unit_word(int u, int total, const Phase& p0, const Phase& p1, const Groups& gr, int G) {
  return u < total ? pack_unit(decode_unit(u, p0, p1, gr, G)) : make_int4(-1, 0, 0, 0);
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded wait until *p >= target (another CTA's release).  False on timeout or abort.
__device__ __noinline__ bool wait_count(const int* p, int target, volatile int* abort_flag) {
  unsigned long long t0 = 0;
  for (uint32_t it = 1;; ++it) {
    if (ld_acquire(p) >= target) return true;
    if ((it & 15u) == 0) {
      if (*abort_flag) return false;
      const unsigned long long now = globaltimer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitNs) return false;
    }
  }
}

// A warp's 32 features of the 32 token columns from column c (the ones past
// c_hi are not stored): round, transpose, store 64 contiguous bytes of 8 token
// rows at a time.  Phase 0 (p) applies GELU and writes rows row0 + column;
// phase 1 scatters to rows dr (32 tokens per register from c_lo on; -1: none).
// `base` is this lane's 8 features of row 0.
template <bool TANH>
__device__ __forceinline__ void store32(uint32_t* v, int c, int c_lo, int c_hi, int p, int row0, const int4& dr,
                                        __nv_bfloat16* base, int N, uint32_t* stage) {
  const int lane = threadIdx.x & 31, st_tok = lane >> 2;
  if (p == 0) {
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      const float z = __uint_as_float(v[q]);
      v[q] = __float_as_uint(TANH ? gelu_tanh_hw(z) : gelu_f(z, 0));
    }
  }
  __syncwarp();
  stage_by_token(stage, lane, [&](int t) { return __uint_as_float(v[t]); });
  __syncwarp();
  const int src = (c - c_lo) >> 5;
  const int d = src == 0 ? dr.x : (src == 1 ? dr.y : (src == 2 ? dr.z : dr.w));
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int tok = it * 8 + st_tok;
    const uint4 val = *reinterpret_cast<const uint4*>(stage + tok * 16 + (lane & 3) * 4);
    const int dl = __shfl_sync(0xffffffffu, d, tok);
    const int row = p == 0 ? row0 + c + tok : dl;
    if (c + tok < c_hi && row >= 0) *reinterpret_cast<uint4*>(base + static_cast<size_t>(row) * N) = val;
  }
}

// A warp's part of a finished tile, columns [c_lo, c_hi), from TMEM to memory,
// 32 columns at a time (each chunk's load is waited for: the eight warps of a
// CTA hide it for each other).
template <bool TANH>
__device__ __forceinline__ void store_tile(uint32_t tb, int c_lo, int c_hi, int p, int row0, int4 dr, __nv_bfloat16* base,
                                        int N, uint32_t* stage) {
#pragma unroll 1
  for (int c = c_lo; c < c_hi; c += 32) {
    uint32_t v[32];
    tmem_ld32_async(tb + c, v);
    tmem_wait32(v);
    store32<TANH>(v, c, c_lo, c_hi, p, row0, dr, base, N, stage);
  }
}

template <bool TANH>
__global__ void __launch_bounds__(kThreads, 1)
    ffn_tc_kernel(const __grid_constant__ TcMapPair maps, const TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];   // leader's: the stage's bytes of both CTAs
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t tfull_bar[2];
  __shared__ __align__(8) uint64_t tempty_bar[2];          // leader's: the epilogue warps of both CTAs
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ __align__(8) uint64_t uq_full[kUQ];
  __shared__ __align__(8) uint64_t uq_empty[kUQ];          // leader's
  __shared__ __align__(16) int4 uq[kUQ];
  __shared__ __align__(8) uint64_t pub_bar[kUQ];           // the epilogue warps' stores of a phase-1 unit are done
  __shared__ uint32_t tmem_base_sh;
  __shared__ Groups gr;
  __shared__ int nmax_sh;
  __shared__ int ticket_sh;  // leader's: the pair's first ticket
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = a.G;
  const uint32_t rank = cluster_rank();

  // Everything that does not read the previous kernel's output happens
  // before the programmatic-dependency wait: barriers, TMEM, map prefetch.
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
    for (int q = 0; q < kUQ; ++q) {
      mbar_init(smem_u32(&uq_full[q]), 1);
      mbar_init(smem_u32(&pub_bar[q]), kEpiWarps);
      // Both CTAs' token producer, epilogue warps and publisher, the MMA
      // thread, the peer's weight producer.
      mbar_init(smem_u32(&uq_empty[q]), 2 * (1 + kEpiWarps + 1) + 2);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_base_sh)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    tc_fence_before();
    // The pair's first ticket.  The counter was re-armed by a combine that lies
    // before the previous kernel, which has passed its own wait.
    if (lane == 0 && rank == 0) ticket_sh = atomicAdd(a.work, 1);
  }
  if (warp == 2 && lane < 2 * (kBoxes + 2)) {
    const TcMaps& m = maps.p[lane & 1];
    const int j = lane >> 1;
    const CUtensorMap* t = j == 0 ? &m.w : (j == 1 ? &m.ws : &m.act[j - 2]);
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(t)) : "memory");
  }
  if (warp == 0) {
    // Bring the launch parameters into the constant cache while the previous
    // kernel finishes (the roles read them right after the wait).
    asm volatile("" ::"r"(a.N[0]), "r"(a.N[1]), "r"(a.K[0]), "r"(a.K[1]), "r"(a.cap), "r"(a.split), "r"(a.units_max),
                 "l"(a.counts), "l"(a.offsets), "l"(a.list), "l"(a.hmid), "l"(a.dep), "l"(a.cache_h), "l"(a.work),
                 "r"(a.E), "r"(a.dep_pairs));
  }
  cluster_arrive();
  cluster_wait();  // both CTAs' barriers are initialised, the leader has its ticket
  // The weight producers' next unit (after the first, the leader's alone).  The
  // draw and its way to the peer lie before the dependency wait (code that runs
  // first after it is fetched while the weights stream in: an mbarrier or the
  // unit queue there cost 1.2 us a launch), and the draw follows the TMEM
  // allocation (drawn by other warps it cost 0.5 to 2 us).  So placed it costs
  // nothing against first units fixed to the pair's index (12-layer D 768 stack
  // 0.747 -> 0.748 ms a step; one layer of it, four steps, 279 -> 278 us).
  int ticket = 0;
  if (threadIdx.x == 0) ticket = ld_cluster(cluster_addr(smem_u32(&ticket_sh), 0));
  Phase p0, p1;
  p0.nw = (a.N[0] + 255) >> 8;
  p1.nw = (a.N[1] + 255) >> 8;
  p0.sub = a.K[0] / kBK;
  p1.sub = a.K[1] / kBK;
  p0.ks = (p0.sub + kSub - 1) / kSub;
  p1.ks = (p1.sub + kSub - 1) / kSub;
  p0.S = p1.S = 1;
  pdl_entry();
  if (warp == 0) {
    // Group sizes, loaded by all lanes at once: each group's token tiles (as
    // few as the cap allows, of equal width) and the tiles ahead of it.
    int tiles = 0, nmax = 32;
    for (int g0 = 0; g0 < G; g0 += 32) {
      const int g = g0 + lane;
      const int c = g < G ? a.counts[g] : 0;
      const int o = g < G ? a.offsets[g] : 0;
      const int nt = (c + a.cap - 1) / a.cap;
      const int wid = nt ? ((c + nt - 1) / nt + 31) & ~31 : 32;
      int incl = nt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
      }
      if (g < G) {
        gr.cnt[g] = c;
        gr.off[g] = o;
        gr.wid[g] = wid;
        gr.before[g] = tiles + incl - nt;
      }
      tiles += __shfl_sync(0xffffffffu, incl, 31);
      nmax = max(nmax, __reduce_max_sync(0xffffffffu, wid));
    }
    if (lane == 0) {
      gr.before[G] = tiles;
      nmax_sh = nmax;
      if (tiles > a.dep_pairs) {
        report_status(a.status, kStatusBadIndex, 5000000 + tiles);
        abort_flag = 1;
      }
    }
  }
  // The group tables are warp 0's; it goes on without waiting for the others.
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const int tiles = gr.before[G];
  // Forced K splits of phase 2, while each split has a stage and the workspace holds the units.
  p1.S = a.split > 1 && p1.ks >= a.split && tiles * p1.nw * a.split <= a.units_max ? a.split : 1;
  p0.units = tiles * p0.nw;
  p1.units = tiles * p1.nw * p1.S;
  const int total = abort_flag ? 0 : p0.units + p1.units;
  // One ring for both phases: slots sized for the widest token tile.  The
  // roles walk it with running addresses.
  const int slot_bytes = kSub * (kABytes + nmax_sh / 2 * (kBK * 2));
  const int nst = min(kMaxStages, kRingBytes / slot_bytes);
  const int dep_target = 2 * p0.nw;
  const uint32_t ring = smem_u32(smem), ring_end = ring + nst * slot_bytes;
  const uint32_t empty0 = smem_u32(&empty_bar[0]);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- Weight producer ----------------
      const bool leader = rank == 0;
      uint32_t dst = ring, eb = empty0;  // the current slot and its barriers
      uint32_t par = 1u;                 // parity its release is waited for with
      int issued = 0;
      bool ok = true;
      int qs = 0;
      uint32_t qpar = 0u;
      const uint32_t full0 = cluster_addr(smem_u32(&full_bar[0]), 0);
      uint32_t fb = full0;
      const uint32_t uqe0 = cluster_addr(smem_u32(&uq_empty[0]), 0);
      const uint32_t uqf1 = cluster_addr(smem_u32(&uq_full[0]), 1);
      const uint32_t uq1 = cluster_addr(smem_u32(&uq[0]), 1);
      // Units: tickets from the shared counter, in increasing order (so phase 1
      // before phase 2 here too).  A pair owns a unit only by drawing it, the
      // first one included: a pair that another stream's kernels keep off the
      // GPU holds up nobody's phase 2.  The leader decodes each unit and passes
      // it to the other roles of both CTAs through the unit queue; a negative
      // word ends it.  The next ticket is drawn four stages before the end of a
      // unit and passed on one stage before it, so that neither round trip
      // leaves the ring idle.
      auto push = [&](const int4& v) -> bool {
        if (!mbar_wait(smem_u32(&uq_empty[qs]), qpar ^ 1u, &abort_flag)) return false;
        uq[qs] = v;
        st_cluster(uq1 + qs * 16, v);
        mbar_arrive(smem_u32(&uq_full[qs]));
        mbar_arrive_cluster(uqf1 + qs * 8);
        if (++qs == kUQ) {
          qs = 0;
          qpar ^= 1u;
        }
        return true;
      };
      // The first unit does without the queue: both CTAs have its ticket.
      int4 cur = unit_word(ticket, total, p0, p1, gr, G);
      if (leader) ok = push(cur);
      for (bool first = true; ok; first = false) {
        if (!leader) {
          if (!first) {
            if (!(ok = mbar_wait_cluster(smem_u32(&uq_full[qs]), qpar, &abort_flag))) break;
            cur = uq[qs];
          }
          mbar_arrive_cluster(uqe0 + qs * 8);
          if (++qs == kUQ) {
            qs = 0;
            qpar ^= 1u;
          }
        }
        if (cur.x < 0) break;
        const Unit t = unpack_unit(cur);
        const TcMaps& mp = maps.p[t.p];
        const int ks = t.p ? p1.ks : p0.ks, S = t.p ? p1.S : p0.S, N = a.N[t.p];
        const CUtensorMap* tw = t.g < a.E ? &mp.w : &mp.ws;
        const int feat = t.w * 256 + static_cast<int>(rank) * kBM;
        // A half tile without weight rows is copied from past the map's last row
        // (zeros, no traffic): a CTA that brought nothing could be lapped by the
        // MMAs, and a barrier two phases on looks like one not yet completed.
        const int wrow = feat < N ? (t.g < a.E ? t.g * N : 0) + feat : (t.g < a.E ? a.E * N : N);
        const int k0 = t.sp * ks / S, k1 = (t.sp + 1) * ks / S;  // stages of this unit
        // Bytes a stage brings into both CTAs (sub-blocks past the last are zero-filled).
        const uint32_t stage_tx = kSub * (2 * kABytes + t.n * (kBK * 2));
        int k = k0;
        for (int part = 0; part < 3 && ok; ++part) {
          // Up to four stages before the end, up to one, to the end.
          const int to = part == 0 ? max(k0, k1 - 4) : (part == 1 ? k1 - 1 : k1);
          for (; k < to; ++k) {
            // The slot is free in both CTAs once the MMAs that read it are
            // done; the leader arms its barrier with the bytes of both CTAs.
            if (!(ok = mbar_wait_hot(eb, par, &abort_flag))) break;
            if (leader) mbar_expect_tx(fb, stage_tx);
            tma_load_k64_pair(dst, tw, wrow, k * kSub, fb);
            ++issued;
            dst += slot_bytes;
            eb += 8;
            fb += 8;
            if (dst == ring_end) {
              dst = ring;
              eb = empty0;
              fb = full0;
              par ^= 1u;
            }
          }
          if (leader && ok) {
            if (part == 0) ticket = atomicAdd(a.work, 1);
            if (part == 1) {
              cur = unit_word(ticket, total, p0, p1, gr, G);
              ok = push(cur);
            }
          }
        }
      }
      if (!ok) {
        if (!abort_flag) report_status(a.status, kStatusWaitTimeout, 101);
        abort_flag = 1;
        // Let the copies already issued land before the CTAs can exit: wait
        // for the newest use of every slot (the leader's barriers see both CTAs').
        for (int q = 0; leader && q < nst && q < issued; ++q) {
          const int last = issued - 1 - (issued - 1 - q) % nst;
          const unsigned long long t0 = globaltimer();
          while (!mbar_try(smem_u32(&full_bar[q]), (last / nst) & 1) && globaltimer() - t0 < kWaitNs) {
          }
        }
      }
    }
  } else if (warp == kTokWarp) {
    if (lane == 0) {
      // ---------------- Token producer ----------------
      const uint32_t ring_t = ring + kSub * kABytes;  // the token half of the first slot
      uint32_t dst = ring_t, eb = empty0;
      uint32_t par = 1u;
      bool ok = true;
      int qs = 0;
      uint32_t qpar = 0u;
      const uint32_t full0 = cluster_addr(smem_u32(&full_bar[0]), 0);
      uint32_t fb = full0;
      const uint32_t uqe0 = cluster_addr(smem_u32(&uq_empty[0]), 0);
      for (;;) {
        if (!(ok = mbar_wait_cluster(smem_u32(&uq_full[qs]), qpar, &abort_flag))) break;
        const int4 cur = uq[qs];
        mbar_arrive_cluster(uqe0 + qs * 8);
        if (++qs == kUQ) {
          qs = 0;
          qpar ^= 1u;
        }
        if (cur.x < 0) break;
        const Unit t = unpack_unit(cur);
        const int ks = t.p ? p1.ks : p0.ks, S = t.p ? p1.S : p0.S;
        const CUtensorMap* ta = &maps.p[t.p].act[(t.n >> 5) - 1];
        const int arow = t.row0 + static_cast<int>(rank) * (t.n >> 1);
        const int k0 = t.sp * ks / S, k1 = (t.sp + 1) * ks / S;
        if (t.p == 1) {
          // The tile's hidden rows come from every phase-1 tile of its rows,
          // stored by other CTAs' epilogues with generic stores and read here
          // by TMA.
          int* d = a.dep + 2 * t.tt;
          if (!(ok = wait_count(d, dep_target, &abort_flag))) break;
          asm volatile("fence.proxy.async.global;" ::: "memory");
          // The last phase-2 CTA to start on this token tile re-arms its counters.
          if (atomicAdd(d + 1, 1) == 2 * p1.nw * S - 1) {
            d[0] = 0;
            d[1] = 0;
          }
        }
        for (int k = k0; k < k1; ++k) {
          if (!(ok = mbar_wait_hot(eb, par, &abort_flag))) break;
          tma_load_k64_pair(dst, ta, arow, k * kSub, fb);
          dst += slot_bytes;
          eb += 8;
          fb += 8;
          if (dst - kSub * kABytes == ring_end) {
            dst = ring_t;
            eb = empty0;
            fb = full0;
            par ^= 1u;
          }
        }
      }
      if (!ok) {
        if (!abort_flag) report_status(a.status, kStatusWaitTimeout, 102);
        abort_flag = 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // ---------------- MMA issuer (the leader, for both CTAs) ----------------
      // Low descriptor words of the current slot's operands (addresses in
      // 16-byte units; smem_desc's leading offset field set).
      const uint32_t w_lo0 = ((ring & 0x3FFFFu) >> 4) | (1u << 16), slot_lo = static_cast<uint32_t>(slot_bytes) >> 4;
      const uint32_t w_end = w_lo0 + nst * slot_lo;
      const uint32_t full0 = smem_u32(&full_bar[0]);
      uint32_t w_lo = w_lo0, fb = full0, eb = empty0;
      uint32_t par = 0u;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      int qs = 0;
      uint32_t qpar = 0u;
      for (;;) {
        if (!(ok = mbar_wait(smem_u32(&uq_full[qs]), qpar, &abort_flag))) break;
        const int4 cur = uq[qs];
        mbar_arrive(smem_u32(&uq_empty[qs]));
        if (++qs == kUQ) {
          qs = 0;
          qpar ^= 1u;
        }
        if (cur.x < 0) break;
        const Unit t = unpack_unit(cur);
        const int ks = t.p ? p1.ks : p0.ks, S = t.p ? p1.S : p0.S;
        const int k0 = t.sp * ks / S, k1 = (t.sp + 1) * ks / S;
        const int n = t.n, sub = t.p ? p1.sub : p0.sub;
        const uint32_t idesc = instr_desc(2 * kBM, n);
        const uint32_t b_sub = n * kBK >> 4;  // a token sub-block in one CTA: n / 2 rows of 128 bytes
        if (!(ok = mbar_wait(smem_u32(&tempty_bar[acc]), acc_phase ^ 1u, &abort_flag))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + static_cast<uint32_t>(acc * kMaxN);
        for (int k = k0; k < k1; ++k) {
          if (!(ok = mbar_wait_hot(fb, par, &abort_flag))) break;
          tc_fence_after();
#pragma unroll
          for (int q = 0; q < kSub; ++q) {
            if (q && k * kSub + q >= sub) break;
            const uint32_t wq = w_lo + q * (kABytes >> 4), xq = w_lo + (kSub * kABytes >> 4) + q * b_sub;
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              mma_bf16_pair(d_tmem, wq + kk * 2, xq + kk * 2, idesc, k != k0 || q != 0 || kk != 0);
          }
          mma_commit_pair(eb);
          w_lo += slot_lo;
          fb += 8;
          eb += 8;
          if (w_lo == w_end) {
            w_lo = w_lo0;
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
        if (!abort_flag) report_status(a.status, kStatusWaitTimeout, 201);
        abort_flag = 1;
      }
      // Every MMA this thread issued has completed once the drain barrier fires.
      mma_commit_pair(smem_u32(&drain_bar), 1);
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(smem_u32(&drain_bar), 0) && globaltimer() - t0 < kWaitNs) {
      }
    }
  } else if (warp == kPubWarp) {
    if (lane == 0) {
      // ---------------- Publisher ----------------
      // The hidden rows of a stored half tile are read by the phase-2 units of
      // its token tile through the async (TMA) proxy: every writer ordered its
      // stores before later async-proxy accesses, the barrier collects the
      // epilogue's warps, and one release add makes them visible with the count.
      const uint32_t uqe0 = cluster_addr(smem_u32(&uq_empty[0]), 0);
      int qs = 0;
      uint32_t qpar = 0u, ppar = 0u;  // ppar bit q: parity of pub_bar[q]
      for (;;) {
        if (!mbar_wait_cluster(smem_u32(&uq_full[qs]), qpar, &abort_flag)) break;
        const int4 cur = uq[qs];
        if (cur.x >= 0 && !(cur.x & 1)) {
          if (!mbar_wait(smem_u32(&pub_bar[qs]), (ppar >> qs) & 1u, &abort_flag)) break;
          ppar ^= 1u << qs;
          asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.dep + 2 * cur.y) : "memory");
        }
        mbar_arrive_cluster(uqe0 + qs * 8);
        if (++qs == kUQ) {
          qs = 0;
          qpar ^= 1u;
        }
        if (cur.x < 0) break;
      }
    }
  } else {
    // ---------------- Epilogue ----------------
    // The warps run independently of each other.
    uint32_t* stage = reinterpret_cast<uint32_t*>(smem + kRingBytes + (warp - 2) * kStageOut);
    const int quad = warp & 3;         // TMEM lanes [32 quad, 32 quad + 32)
    const int half = (warp - 2) >> 2;  // which half of the tile's token columns
    const uint32_t uqe0 = cluster_addr(smem_u32(&uq_empty[0]), 0);
    const uint32_t tempty0 = cluster_addr(smem_u32(&tempty_bar[0]), 0);
    int acc = 0;
    uint32_t acc_phase = 0;
    int qs = 0;
    uint32_t qpar = 0u;
    bool ok;
    for (;;) {
      if (!(ok = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&uq_full[qs]), qpar, &abort_flag)))) break;
      const int4 cur = uq[qs];
      const uint32_t pub = smem_u32(&pub_bar[qs]);
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(uqe0 + qs * 8);
      if (++qs == kUQ) {
        qs = 0;
        qpar ^= 1u;
      }
      if (cur.x < 0) break;
      const Unit t = unpack_unit(cur);
      const int S = t.p ? p1.S : p0.S, N = a.N[t.p];
      const int feat = t.w * 256 + static_cast<int>(rank) * kBM + quad * 32;  // the warp's 32 features
      // The warp's token columns (none if it has no features).
      const int c_lo = half * (t.n >> 1), c_hi = feat < N ? min(c_lo + (t.n >> 1), t.valid) : 0;
      // Phase 2: the destination rows of the warp's tokens, 32 per register
      // (loaded while the MMAs run).
      int4 dr = make_int4(-1, -1, -1, -1);
      if (t.p == 1) {
        const int lim = t.g < a.E ? a.T * a.k : a.T;
        auto dest = [&](int c) -> int {
          if (c >= c_hi) return -1;
          const int d = a.list[t.row0 + c];
          if (d >= 0 && d < lim) return d;
          report_status(a.status, kStatusBadIndex, 4000000 + t.row0 + c);
          return -1;
        };
        dr = make_int4(dest(c_lo + lane), dest(c_lo + 32 + lane), dest(c_lo + 64 + lane), dest(c_lo + 96 + lane));
      }
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&tfull_bar[acc]), acc_phase, &abort_flag)))) break;
      tc_fence_after();
      __nv_bfloat16* base = static_cast<__nv_bfloat16*>(t.p == 0 ? a.hmid : (t.g < a.E ? a.cache_h : a.shared_h)) +
                            feat + (lane & 3) * 8;
      const uint32_t tb = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(acc * kMaxN);
      if (S == 1) {
        if (c_lo < c_hi) store_tile<TANH>(tb, c_lo, c_hi, t.p, t.row0, dr, base, N, stage);
        if (t.p == 0) asm volatile("fence.proxy.async.global;" ::: "memory");  // see the publisher
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_cluster(tempty0 + acc * 8);
          if (t.p == 0) mbar_arrive(pub);
        }
      } else {
        // Split K: park this split's fp32 columns ([token column][128
        // features], so each access covers 128 contiguous bytes), free TMEM,
        // then the last split to arrive for the warp's part of the tile sums
        // the splits in split order.
        const int tile = 2 * (t.tt * p1.nw + t.w) + static_cast<int>(rank);
        const size_t slice = static_cast<size_t>(kBM) * kMaxN;
        float* parked = a.partial + static_cast<size_t>(tile) * S * slice + quad * 32 + lane;
        for (int c = c_lo; c < c_hi; c += 32) {
          uint32_t v[32];
          tmem_ld32_async(tb + c, v);
          tmem_wait32(v);
#pragma unroll
          for (int q = 0; q < 32; ++q)
            if (c + q < c_hi) parked[t.sp * slice + (c + q) * kBM] = __uint_as_float(v[q]);
        }
        tc_fence_before();
        __threadfence();
        __syncwarp();
        int arrived = 0;
        int* sem = a.tile_sem + tile * kEpiWarps + (warp - 2);
        if (lane == 0) {
          mbar_arrive_cluster(tempty0 + acc * 8);
          arrived = atomicAdd(sem, 1);
        }
        if (__shfl_sync(0xffffffffu, arrived, 0) == S - 1) {
          __threadfence();
          for (int c = c_lo; c < c_hi; c += 32) {
            // One split's 32 values in flight at a time, added in split order.
            float sum[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) sum[q] = c + q < c_hi ? __ldcg(parked + (c + q) * kBM) : 0.f;
            for (int z = 1; z < S; ++z) {
              float f[32];
#pragma unroll
              for (int q = 0; q < 32; ++q) f[q] = c + q < c_hi ? __ldcg(parked + z * slice + (c + q) * kBM) : 0.f;
#pragma unroll
              for (int q = 0; q < 32; ++q) sum[q] += f[q];
            }
            uint32_t v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = __float_as_uint(sum[q]);
            store32<TANH>(v, c, c_lo, c_hi, t.p, t.row0, dr, base, N, stage);
          }
          if (lane == 0) *sem = 0;
        }
      }
      if (++acc == 2) {
        acc = 0;
        acc_phase ^= 1u;
      }
    }
    if (!ok) {
      if (lane == 0 && !abort_flag) report_status(a.status, kStatusWaitTimeout, 301);
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

struct TcPlan {
  TcMapPair maps;  // phase 1 (N = F, K = D) and phase 2 (N = D, K = F)
  int cap, split, n_sms, n_pairs;
};

namespace {
size_t split_slices(int n_sms) { return static_cast<size_t>(4) * n_sms; }
}  // namespace
size_t tc_split_sems(int n_sms) { return split_slices(n_sms) * kEpiWarps; }
size_t tc_partial_bytes(int n_sms) { return split_slices(n_sms) * kBM * kMaxN * sizeof(float); }
// Token tiles a launch can have at the narrowest cap (64): every group's rows rounded up.
size_t tc_dep_pairs(int max_rows, int G) { return static_cast<size_t>((max_rows + 63) / 64 + G); }

namespace {

bool encode_phase(TcMaps* m, const void* act, uint64_t rows, uint64_t K, const void* w, uint64_t w_rows,
                  const void* ws, uint64_t ws_rows) {
  if (!encode_k64(&m->w, w, w_rows, K, kBM, kSub)) return false;
  if (ws) {
    if (!encode_k64(&m->ws, ws, ws_rows, K, kBM, kSub)) return false;
  } else {
    m->ws = m->w;  // never read: there is no shared group
  }
  for (int i = 0; i < kBoxes; ++i)
    if (!encode_k64(&m->act[i], act, rows, K, 16 * (i + 1), kSub)) return false;
  return true;
}

// Pairs that can be resident at once: one CTA per SM, both CTAs of a pair in
// one GPU processing cluster.
template <typename K>
int resident_pairs(K kernel, int n_sms) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_sms / 2 * 2);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return std::min(n, n_sms / 2);
}

}  // namespace

TcPlan* tc_plan_create(const FfnArgs& a, int n_sms, char* err, int errlen) {
  TcPlan* p = new TcPlan();
  p->n_sms = n_sms;
  p->cap = a.tile_n ? a.tile_n : kMaxN;
  p->split = a.split_k;
  const char* what = nullptr;
  if (a.D % kBK || a.F % kBK) what = "hidden and ffn must be multiples of 64";
  else if (!get_encoder()) what = "cuTensorMapEncodeTiled is unavailable";
  else if (!encode_phase(&p->maps.p[0], a.xg, a.max_rows, a.D, a.w1, static_cast<uint64_t>(a.E) * a.F, a.ws1, a.F) ||
           !encode_phase(&p->maps.p[1], a.hmid, a.max_rows, a.F, a.w2, static_cast<uint64_t>(a.E) * a.D, a.ws2, a.D))
    what = "tensor map encoding failed";
  auto reserve = [&](auto kernel) {
    if (set_dyn_smem_on_device(reinterpret_cast<const void*>(kernel), kSmemBytes) != cudaSuccess) {
      cudaGetLastError();
      what = "cannot reserve shared memory for the tensor-core kernel";
      return;
    }
    p->n_pairs = resident_pairs(kernel, n_sms);
    if (p->n_pairs < 1) what = "no CTA pair of the tensor-core kernel fits the device";
  };
  if (!what) {
    if (a.gelu_tanh) reserve(ffn_tc_kernel<true>);
    else reserve(ffn_tc_kernel<false>);
  }
  if (what) {
    if (err && errlen > 0) snprintf(err, errlen, "%s", what);
    tc_plan_destroy(p);
    return nullptr;
  }
  return p;
}

void tc_plan_destroy(TcPlan* p) { delete p; }

cudaError_t launch_ffn_tc(TcPlan* p, const FfnArgs& a, cudaStream_t s) {
  TcArgs t{};
  t.G = a.G;
  t.E = a.E;
  t.k = a.k;
  t.T = a.T;
  t.N[0] = t.K[1] = a.F;
  t.N[1] = t.K[0] = a.D;
  t.cap = p->cap;
  t.split = p->split;
  t.units_max = static_cast<int>(split_slices(p->n_sms) / 2);  // two CTAs' slices per unit
  t.counts = a.counts;
  t.offsets = a.offsets;
  t.list = a.list;
  t.hmid = a.hmid;
  t.cache_h = a.cache_h;
  t.shared_h = a.shared_h;
  t.partial = a.partial;
  t.tile_sem = a.tile_sem;
  t.dep = a.dep;
  t.dep_pairs = a.dep_pairs;
  t.work = a.work;
  t.status = a.status;
  const dim3 grid(2 * p->n_pairs);
  return a.gelu_tanh ? launch_pdl<2>(ffn_tc_kernel<true>, grid, dim3(kThreads), kSmemBytes, s, p->maps, t)
                     : launch_pdl<2>(ffn_tc_kernel<false>, grid, dim3(kThreads), kSmemBytes, s, p->maps, t);
}

}  // namespace moeca

// Branch selection and compaction of the branch-cached MoE layer.
//
// select_kernel, one token per thread (Sec. 4.2):
//   * match each routed branch p against the token's cached branches by
//     expert id; an unmatched branch is always recomputed;
//   * score a matched branch  s = w_p + lambda1 |w_p - w_q^{t0}|
//     + lambda2 ||h_q|| / sum_j ||h_j||   (Eq. 9)  and recompute iff s > tau_e;
//   * matched branches keep their cache slot q(p); unmatched ones take the
//     slots whose expert is no longer routed, ascending p -> ascending q;
//     on a full-computation step every branch is recomputed with slot = p;
//   * write the new cache metadata, token_any = (R_i non-empty, Sec. 4.1) and
//     per-block counts of recomputed rows per expert group (warp ballots).
// The last block scans the per-block counts into per-group row offsets.
//
// compact_kernel, same token blocks: ranks each recomputed row inside its
// group in ascending token order (ballot + popc prefix) and writes the row
// list (token * k + slot for routed experts, token for the shared expert).
// gather_kernel then copies every listed row's layer input into a
// contiguous buffer for the GEMMs, one warp per row over the whole list.
//
// decide_kernel does all of it in one launch while its grid of 32-token blocks
// is co-resident (decide_blocks): decisions, an exchange of the blocks' row
// counts, row lists and row gather, as the fused preparation kernel does after
// its thresholds.  The three kernels above take larger token counts.
#include "common.cuh"
#include "exchange.cuh"
#include "kernels.h"
#include "select_token.cuh"

namespace moeca {
namespace {

constexpr int kThreads = kSelectTokensPerBlock;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxGroups = kMaxExperts + 1;

// KMAX >= k bounds the per-token loops at compile time.
template <int KMAX>
__global__ void __launch_bounds__(kThreads) select_kernel(SelectArgs a) {
  pdl_entry();
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int i = blockIdx.x * kThreads + t;
  const bool valid = i < a.T;
  const int k = a.k, E = a.E, G = a.G;
  TokenDecisionT<KMAX> d;
  const size_t b0 = static_cast<size_t>(valid ? i : 0) * a.k;
  decide_token<KMAX>(a, i, valid, a.route_e + b0, a.route_w + b0, a.cache_e + b0, a.cache_w + b0, a.cache_norm + b0, d);
  const int* e = d.e;
  const bool* rec = d.rec;
  const bool any = d.any, bad = d.bad, shared_row = d.shared_row;
  const int n_matched = d.n_matched, n_rec = d.n_rec, n_near = d.n_near;

  // Rows per (warp, group) by ballot, then per block.
  __shared__ int sm_wc[kWarps][kMaxGroups];
  for (int g = 0; g < G; ++g) {
    bool has = false;
    if (g < E) {
#pragma unroll
      for (int p = 0; p < KMAX; ++p) has |= (rec[p] && e[p] == g);
    } else {
      has = shared_row;
    }
    const unsigned b = __ballot_sync(0xffffffffu, has);
    if (lane == 0) sm_wc[warp][g] = __popc(b);
  }
  // Branch counters.
  const int c_matched = warp_sum_i(n_matched);
  const int c_rec = warp_sum_i(n_rec);
  const int c_near = warp_sum_i(n_near);
  const int c_full = warp_sum_i(valid && !bad && !any ? 1 : 0);
  const int c_shared = warp_sum_i(shared_row ? 1 : 0);
  __shared__ int sm_c[kWarps][5];
  if (lane == 0) {
    sm_c[warp][0] = c_matched;
    sm_c[warp][1] = c_rec;
    sm_c[warp][2] = c_near;
    sm_c[warp][3] = c_full;
    sm_c[warp][4] = c_shared;
  }
  __syncthreads();
  for (int g = t; g < G; g += kThreads) {
    int s = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += sm_wc[w][g];
    a.block_counts[static_cast<size_t>(blockIdx.x) * G + g] = s;
  }
  if (t == 0) {
    int tot[5] = {0, 0, 0, 0, 0};
    for (int w = 0; w < kWarps; ++w)
      for (int j = 0; j < 5; ++j) tot[j] += sm_c[w][j];
    const int nb = min(kThreads, a.T - static_cast<int>(blockIdx.x) * kThreads);
    unsigned long long* st = a.stats;
    atomicAdd(st + kStRecomputed, static_cast<unsigned long long>(tot[1]));
    atomicAdd(st + kStReused, static_cast<unsigned long long>(nb * k - tot[1]));
    if (tot[4]) atomicAdd(st + kStSharedRecomputed, static_cast<unsigned long long>(tot[4]));
    if (!a.refresh) {
      atomicAdd(st + kStMatched, static_cast<unsigned long long>(tot[0]));
      atomicAdd(st + kStTokensFullyReused, static_cast<unsigned long long>(tot[3]));
      if (tot[2]) atomicAdd(st + kStNearScore, static_cast<unsigned long long>(tot[2]));
    }
    if (blockIdx.x == 0) {
      const unsigned long long br = static_cast<unsigned long long>(a.T) * k;
      atomicAdd(st + kStLayerSteps, 1ull);
      atomicAdd(st + kStBranches, br);
      if (a.refresh) atomicAdd(st + kStRefreshSteps, 1ull);
      else atomicAdd(st + kStCacheBranches, br);
    }
  }
  // The last block turns per-block counts into offsets.
  __threadfence();
  __syncthreads();
  __shared__ unsigned ticket;
  if (t == 0) ticket = atomicAdd(a.done, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  // Chunks of 16 blocks: every thread loads counts in parallel, then one
  // thread per group scans the chunk in block order.
  __shared__ int sm_tot[kMaxGroups];
  __shared__ int sm_chunk[16][kMaxGroups];
  for (int g = t; g < G; g += kThreads) sm_tot[g] = 0;
  for (unsigned b0 = 0; b0 < gridDim.x; b0 += 16) {
    const int nb = min(16u, gridDim.x - b0);
    __syncthreads();
    for (int idx = t; idx < nb * G; idx += kThreads)
      sm_chunk[idx / G][idx % G] = __ldcg(a.block_counts + static_cast<size_t>(b0 + idx / G) * G + idx % G);
    __syncthreads();
    for (int g = t; g < G; g += kThreads) {
      int run = sm_tot[g];
      for (int j = 0; j < nb; ++j) {
        a.block_offsets[static_cast<size_t>(b0 + j) * G + g] = run;
        run += sm_chunk[j][g];
      }
      sm_tot[g] = run;
    }
  }
  __syncthreads();
  for (int g = t; g < G; g += kThreads) a.counts[g] = sm_tot[g];
  if (t == 0) {
    int off = 0;
    for (int g = 0; g < G; ++g) {
      a.offsets[g] = off;
      off += sm_tot[g];
    }
    a.offsets[G] = off;
    *a.done = 0u;
  }
}

template <typename TI, int KMAX>
__global__ void __launch_bounds__(kThreads) compact_kernel(CompactArgs a) {
  pdl_entry();
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int i = blockIdx.x * kThreads + t;
  const bool valid = i < a.T;
  const int k = a.k, E = a.E, G = a.G;
  int e[KMAX], sl[KMAX];
  bool rec[KMAX];
  bool any = false;
#pragma unroll
  for (int p = 0; p < KMAX; ++p) {
    e[p] = -1;
    sl[p] = 0;
    rec[p] = false;
    if (valid && p < k) {
      const size_t b = static_cast<size_t>(i) * k + p;
      rec[p] = a.recompute[b] != 0;
      e[p] = a.route_e[b];
      sl[p] = a.slot[b];
      if (e[p] < 0 || e[p] >= E) rec[p] = false;  // flagged by select
    }
  }
  if (valid) any = a.token_any[i] != 0;
  const bool shared_row = valid && a.n_shared && (a.refresh || a.shared_policy || any);

  __shared__ unsigned sm_bal[kWarps][kMaxGroups];
  __shared__ int sm_pre[kWarps][kMaxGroups];
  for (int g = 0; g < G; ++g) {
    bool has = false;
    if (g < E) {
#pragma unroll
      for (int p = 0; p < KMAX; ++p) has |= (rec[p] && e[p] == g);
    } else {
      has = shared_row;
    }
    const unsigned b = __ballot_sync(0xffffffffu, has);
    if (lane == 0) sm_bal[warp][g] = b;
  }
  __syncthreads();
  for (int g = t; g < G; g += kThreads) {
    int run = a.offsets[g] + a.block_offsets[static_cast<size_t>(blockIdx.x) * G + g];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      sm_pre[w][g] = run;
      run += __popc(sm_bal[w][g]);
    }
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int p = 0; p < KMAX; ++p) {
    if (rec[p]) {
      const int g = e[p];
      const int pos = sm_pre[warp][g] + __popc(sm_bal[warp][g] & lt);
      a.list[pos] = i * k + sl[p];
    }
  }
  if (shared_row) {
    const int pos = sm_pre[warp][E] + __popc(sm_bal[warp][E] & lt);
    a.list[pos] = i;
  }
}

// Gather of every listed row's layer input into the group-contiguous buffer
// the GEMMs read: one warp per row over the whole list (rows of group g are
// [offsets[g], offsets[g + 1])), 16-byte vectors.  A list entry is
// token * k + slot for a routed group and the token for the shared group.
template <typename TI>
__global__ void __launch_bounds__(256) gather_kernel(CompactArgs a) {
  pdl_entry();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = a.G, E = a.E;
  __shared__ int off_sm[kMaxGroups + 1];  // group offsets, read once
  for (int g = threadIdx.x; g <= G; g += blockDim.x) off_sm[g] = a.offsets[g];
  __syncthreads();
  const int rows = off_sm[G];
  const int nv = a.D * static_cast<int>(sizeof(TI)) / 16;
  const uint4* x = static_cast<const uint4*>(a.x);
  uint4* xg = static_cast<uint4*>(a.xg);
  for (int r = blockIdx.x * 8 + warp; r < rows; r += gridDim.x * 8) {
    // Group of row r: the last g with offsets[g] <= r (G <= 65: a short search).
    int lo = 0, hi = G - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (off_sm[mid] <= r) lo = mid;
      else hi = mid - 1;
    }
    const int ent = a.list[r];
    const int tok = lo < E ? ent / a.k : ent;
    if (tok < 0 || tok >= a.T) {
      if (lane == 0) report_status(a.status, kStatusBadIndex, 5100000 + r);
      continue;
    }
    const uint4* src = x + static_cast<size_t>(tok) * nv;
    uint4* dst = xg + static_cast<size_t>(r) * nv;
    for (int c = lane; c < nv; c += 32) dst[c] = src[c];
  }
}

// ---- select, compact and gather in one launch ----
// The three kernels are latency, not bytes: each starts, waits on a chain of
// loads and ends, with 128 tokens in a block (32 blocks at 4096 tokens), and
// the gather reads a token's row once per recomputed branch.  Here one warp of
// a 32-token block decides a token per lane, the blocks exchange their row
// counts per group as tagged words, and every warp copies its tokens' rows,
// each read once and written to all its places.  Event-timed, three kernels ->
// this one, full / cache step: 64 experts top-8 at 4096 tokens, D 1152
// 42 -> 26 / 36 -> 22 us; D 2560, 4 + 1 experts 29 -> 22 / 25 -> 19 us; fp32,
// D 384, 512 tokens 18 -> 12 us.
constexpr int kDecTokens = 32;
constexpr int kDecThreads = 256;
constexpr unsigned long long kDecWaitNs = 1000000000ull;

template <int KMAX>
__global__ void __launch_bounds__(kDecThreads) decide_kernel(DecideArgs a) {
  __shared__ int32_t s_re[kDecTokens * KMAX], s_ce[kDecTokens * KMAX];
  __shared__ float s_rw[kDecTokens * KMAX], s_cw[kDecTokens * KMAX], s_cn[kDecTokens * KMAX];
  __shared__ float s_tau[kMaxExperts];
  __shared__ unsigned s_bal[kMaxGroups];
  __shared__ int s_part[kDecThreads][2];
  __shared__ int s_pre[kMaxGroups], s_tot[kMaxGroups], s_off[kMaxGroups + 1];
  __shared__ int s_pos[kDecTokens][KMAX + 1];  // list position of each of a token's rows, -1: none
  __shared__ unsigned s_epoch;
  __shared__ int s_fail;
  const SelectArgs& sel = a.sel;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int k = sel.k, E = sel.E, G = sel.G;
  const int tok0 = blockIdx.x * kDecTokens, ntok = min(kDecTokens, sel.T - tok0);
  const size_t b0 = static_cast<size_t>(tok0) * k;
  // Before the dependency wait: the cached metadata.  The previous kernel is
  // this layer's router, which passed its own wait, so the kernels that wrote
  // them (this one and the combine, a step earlier) have ended.
  if (!sel.refresh)
    for (int idx = t; idx < ntok * k; idx += kDecThreads) {
      s_ce[idx] = sel.cache_e[b0 + idx];
      s_cw[idx] = sel.cache_w[b0 + idx];
      s_cn[idx] = sel.cache_norm[b0 + idx];
    }
  pdl_entry();
  // This launch's tag: one past the last launch's, kept on the device (a
  // captured launch can be replayed), and advanced by block 0 once it has read
  // every block's words.  A block publishes after the barrier below, so block 0
  // then knows that every block has read its tag.
  // A launch whose exchange failed leaves the tag as it was or not, and blocks
  // of it may still start: from then on no block publishes, reads words or
  // writes lists, in this launch or a later one (any layer's), until
  // moeca_reset clears the words.  Row counts of different launches under one
  // tag would send list and row writes past their buffers.
  unsigned long long state = 0;  // {epoch, failed}, in flight beside the loads below
  if (t == 0) state = ld_word(reinterpret_cast<const unsigned long long*>(a.state));
  for (int idx = t; idx < ntok * k; idx += kDecThreads) {
    s_re[idx] = sel.route_e[b0 + idx];
    s_rw[idx] = sel.route_w[b0 + idx];
  }
  if (t < E) s_tau[t] = sel.tau[t];
  if (t == 0) {
    const unsigned e = static_cast<unsigned>(state) + 1;
    s_epoch = e ? e : 1;  // 0 marks words never written
    s_fail = static_cast<int>(state >> 32);
  }
  __syncthreads();
  if (s_fail) return;
  const unsigned epoch = s_epoch;

  TokenDecisionT<KMAX> d;
  if (warp == 0) {
    const bool valid = lane < ntok;
    const int q = valid ? lane * k : 0;
    TokenPrepT<KMAX> tp;
    prepare_token(sel, tok0 + lane, valid, s_re + q, s_rw + q, s_ce + q, s_cw + q, s_cn + q, tp);
    finish_token(sel, tok0 + lane, tp, s_tau, d);
    // Groups in which this lane's token has a row.
    uint32_t gm[3] = {0u, 0u, 0u};
#pragma unroll
    for (int p = 0; p < KMAX; ++p)
      if (d.rec[p]) gm[d.e[p] >> 5] |= 1u << (d.e[p] & 31);
    if (d.shared_row) gm[E >> 5] |= 1u << (E & 31);
    for (int g = 0; g < G; ++g) {
      const unsigned b = __ballot_sync(0xffffffffu, (gm[g >> 5] >> (g & 31)) & 1u);
      if (lane == (g & 31)) s_bal[g] = b;
    }
    __syncwarp();
    for (int g = lane; g < G; g += 32)
      st_word(a.words + static_cast<size_t>(blockIdx.x) * G + g, tag_word(__popc(s_bal[g]), epoch));
    const int c_matched = warp_sum_i(d.n_matched), c_rec = warp_sum_i(d.n_rec), c_near = warp_sum_i(d.n_near);
    const int c_full = warp_sum_i(valid && !d.bad && !d.any ? 1 : 0), c_shared = warp_sum_i(d.shared_row ? 1 : 0);
    if (lane == 0) {
      unsigned long long* st = sel.stats;
      atomicAdd(st + kStRecomputed, static_cast<unsigned long long>(c_rec));
      atomicAdd(st + kStReused, static_cast<unsigned long long>(ntok * k - c_rec));
      if (c_shared) atomicAdd(st + kStSharedRecomputed, static_cast<unsigned long long>(c_shared));
      if (!sel.refresh) {
        atomicAdd(st + kStMatched, static_cast<unsigned long long>(c_matched));
        atomicAdd(st + kStTokensFullyReused, static_cast<unsigned long long>(c_full));
        if (c_near) atomicAdd(st + kStNearScore, static_cast<unsigned long long>(c_near));
      }
      if (blockIdx.x == 0) {
        const unsigned long long br = static_cast<unsigned long long>(sel.T) * k;
        atomicAdd(st + kStLayerSteps, 1ull);
        atomicAdd(st + kStBranches, br);
        if (sel.refresh) atomicAdd(st + kStRefreshSteps, 1ull);
        else atomicAdd(st + kStCacheBranches, br);
      }
    }
  }

  // Rows per group of the blocks before this one and of all blocks: a group's
  // blocks in R ranges, one thread each, added in range order.
  {
    const int nb = gridDim.x, me = blockIdx.x;
    const int R = kDecThreads / G, g = t % G, j = t / G;
    int pre = 0, tot = 0;
    bool ok = true;
    if (j < R) {
      const int lo = static_cast<int>(static_cast<long long>(j) * nb / R);
      const int hi = static_cast<int>(static_cast<long long>(j + 1) * nb / R);
      ok = read_tagged<16>(
          a.words, hi - lo, [&](int q) { return static_cast<size_t>(lo + q) * G + g; }, epoch ^ a.stall,
          globaltimer() + kDecWaitNs, [&](int q, uint32_t v) {
            const int c = static_cast<int>(v);
            if (lo + q < me) pre += c;
            tot += c;
          });
    }
    if (!ok) {
      report_status(sel.status, kStatusWaitTimeout, 620);
      *static_cast<volatile unsigned*>(&a.state->failed) = 1u;
      s_fail = 1;
    }
    s_part[t][0] = pre;
    s_part[t][1] = tot;
    __syncthreads();
    if (s_fail) return;
    for (int gg = t; gg < G; gg += kDecThreads) {
      int p2 = 0, t2 = 0;
      for (int jj = 0; jj < R; ++jj) {
        p2 += s_part[jj * G + gg][0];
        t2 += s_part[jj * G + gg][1];
      }
      s_pre[gg] = p2;
      s_tot[gg] = t2;
    }
  }
  __syncthreads();
  if (warp == 0) {
    // Exclusive scan of the group totals into offsets, 32 groups at a time.
    int carry = 0;
    for (int g0 = 0; g0 < G; g0 += 32) {
      const int g = g0 + lane;
      const int v = g < G ? s_tot[g] : 0;
      int incl = v;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, dd);
        if (lane >= dd) incl += u;
      }
      if (g < G) s_off[g] = carry + incl - v;
      carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) s_off[G] = carry;
    __syncwarp();
    // The block's row lists, ascending tokens within each group.
    bool over = false;  // a place past the list's end (its row is left out)
    auto in_list = [&](int pos, int row) {
      const bool in = pos < a.rows;
      over |= !in;
      if (in) a.list[pos] = row;
      return in ? pos : -1;
    };
    const unsigned lt = (1u << lane) - 1u;
    const int i = tok0 + lane;
#pragma unroll
    for (int p = 0; p < KMAX; ++p) {
      int pos = -1;
      if (d.rec[p]) {
        const int g = d.e[p];
        pos = in_list(s_off[g] + s_pre[g] + __popc(s_bal[g] & lt), i * k + d.sl[p]);
      }
      s_pos[lane][p] = pos;
    }
    int pos = -1;
    if (d.shared_row) pos = in_list(s_off[E] + s_pre[E] + __popc(s_bal[E] & lt), i);
    s_pos[lane][KMAX] = pos;
    if (over) report_status(sel.status, kStatusBadIndex, 6200000 + i);
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    if (t == 0) a.state->epoch = epoch;
    for (int g = t; g < G; g += kDecThreads) sel.counts[g] = s_tot[g];
    for (int g = t; g <= G; g += kDecThreads) sel.offsets[g] = s_off[g];
  }
  if (!a.xg) return;
  // One warp per token: its row, read once, to each of its places.
  constexpr int kC = 4;
  const uint4* x = static_cast<const uint4*>(a.x);
  uint4* xg = static_cast<uint4*>(a.xg);
  const int nv = a.row_vecs;
  for (int q = warp; q < ntok; q += kDecThreads / 32) {
    const uint4* src = x + static_cast<size_t>(tok0 + q) * nv;
    for (int c0 = lane; c0 < nv; c0 += 32 * kC) {
      uint4 v[kC];
#pragma unroll
      for (int u = 0; u < kC; ++u)
        if (c0 + 32 * u < nv) v[u] = src[c0 + 32 * u];
#pragma unroll
      for (int p = 0; p <= KMAX; ++p) {
        const int pos = s_pos[q][p];
        if (pos < 0) continue;
        uint4* dst = xg + static_cast<size_t>(pos) * nv;
#pragma unroll
        for (int u = 0; u < kC; ++u)
          if (c0 + 32 * u < nv) dst[c0 + 32 * u] = v[u];
      }
    }
  }
}

template <typename F>
auto with_kmax(int k, F&& f) {
  if (k <= 2) return f(decide_kernel<2>);
  if (k <= 4) return f(decide_kernel<4>);
  return f(decide_kernel<kMaxTopK>);
}

}  // namespace

int decide_blocks(int max_tokens, int k, int n_sms) {
  const int nb = (max_tokens + kDecTokens - 1) / kDecTokens;
  int occ = 0;
  const cudaError_t e = with_kmax(k, [&](auto kern) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kDecThreads, 0);
  });
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  // Two such launches fit at once: the blocks wait for each other, so launches
  // of two streams must not keep each other's blocks off the GPU.  (Room for
  // four, by 64 registers a thread, spilled: top-8 / E 64 650 -> 900 us a pass.)
  return static_cast<long long>(occ) * n_sms >= 2ll * nb ? nb : 0;
}

cudaError_t launch_decide(const DecideArgs& a, cudaStream_t s) {
  const dim3 grid((a.sel.T + kDecTokens - 1) / kDecTokens);
  return with_kmax(a.sel.k, [&](auto kern) { return launch_pdl(kern, grid, dim3(kDecThreads), 0, s, a); });
}

cudaError_t launch_select(const SelectArgs& a, cudaStream_t s) {
  const int grid = (a.T + kThreads - 1) / kThreads;
  if (a.k <= 2) return launch_pdl(select_kernel<2>, dim3(grid), dim3(kThreads), 0, s, a);
  if (a.k <= 4) return launch_pdl(select_kernel<4>, dim3(grid), dim3(kThreads), 0, s, a);
  return launch_pdl(select_kernel<kMaxTopK>, dim3(grid), dim3(kThreads), 0, s, a);
}

cudaError_t launch_compact(const CompactArgs& a, bool bf16, cudaStream_t s) {
  const int grid = (a.T + kThreads - 1) / kThreads;
  auto run = [&](auto kern) { return launch_pdl(kern, dim3(grid), dim3(kThreads), 0, s, a); };
  cudaError_t e;
  if (bf16) e = a.k <= 2 ? run(compact_kernel<__nv_bfloat16, 2>) : a.k <= 4 ? run(compact_kernel<__nv_bfloat16, 4>)
                                                                            : run(compact_kernel<__nv_bfloat16, kMaxTopK>);
  else e = a.k <= 2 ? run(compact_kernel<float, 2>) : a.k <= 4 ? run(compact_kernel<float, 4>)
                                                             : run(compact_kernel<float, kMaxTopK>);
  if (e != cudaSuccess || a.xg == nullptr) return e;
  // The row gather runs over the whole list, one warp per row.
  const int rows = a.T * (a.k + a.n_shared);
  const int ggrid = (rows + 7) / 8;
  return bf16 ? launch_pdl(gather_kernel<__nv_bfloat16>, dim3(ggrid), dim3(256), 0, s, a)
              : launch_pdl(gather_kernel<float>, dim3(ggrid), dim3(256), 0, s, a);
}

cudaError_t launch_gather(const CompactArgs& a, bool bf16, cudaStream_t s) {
  const int rows = a.T * (a.k + a.n_shared);
  const int ggrid = (rows + 7) / 8;
  return bf16 ? launch_pdl(gather_kernel<__nv_bfloat16>, dim3(ggrid), dim3(256), 0, s, a)
              : launch_pdl(gather_kernel<float>, dim3(ggrid), dim3(256), 0, s, a);
}

}  // namespace moeca

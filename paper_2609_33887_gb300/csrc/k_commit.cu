// Merge of the per-part softmax partials and the threshold commit with the
// per-block top-1 fallback, for every tau of the grid in one pass.
//
// One CTA of 32 warps per block of the window. A thread takes one position and
// every 32nd (blocks longer than 32: every 16th) partial slot, its loads issued
// together; a warp then merges a position's (or two positions') threads by
// shuffles, and warp 0 applies, for every tau_k, the rule
//   commit(p, k) = masked(p) && active(block) && conf(p) >= tau_k           (Sec. 3.1, App. B.1)
//                  || the block is fallback-eligible, holds a masked position,
//                     no position cleared tau_k, and p is the masked position of
//                     highest confidence (lowest position on ties)         (App. B.2)
// with one warp ballot per tau (two for blocks longer than 32).
//
// Vocabulary-parallel split (one head shard per rank): MERGE_EMIT merges the
// slots of each position of this shard's LM head into one partial per window
// position (global token ids: the shard's offset added) instead of
// committing; MERGE_GATHERED merges the n_parts such per-position partials
// gathered from every shard ([n_parts, P] arrays) and commits.
#include "checks.h"
#include "kernels.h"

namespace bd {

namespace {
constexpr int THREADS = 1024;
constexpr int MAX_L = 64;
// Partial slots a thread loads at once. The kernel's bound is its chain of
// latencies (header, row, partials, combines): it ends 3.8 us after the LM head
// on the 8 x 2 x 32 window, 5.5 us with 256 threads that took nine slots each
// and warp 0 merging eight groups per position.
constexpr int BATCH = 4;
}  // namespace

// LP: positions a CTA handles side by side, 32 or 64 (>= the block length)
template <int MODE, int LP>
__global__ void __launch_bounds__(THREADS) merge_commit_kernel(CommitArgs a) {
  constexpr int GROUPS = THREADS / LP;  // threads per position
  // thread (group g, position j): [j][g], padded so that both directions hit different banks
  __shared__ float sm_m[LP][GROUPS + 1], sm_s[LP][GROUPS + 1];
  __shared__ int sm_a[LP][GROUPS + 1];
  // the merged state of each position, and whether it has a compacted row
  __shared__ float mg_m[LP], mg_s[LP];
  __shared__ int mg_a[LP];
  __shared__ bool sm_live[LP];
  const int blk = blockIdx.x;
  const int L = a.block_len;
  const int64_t base = static_cast<int64_t>(blk) * L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_launch_dependents();  // a kernel behind this one waits for it before touching memory
  griddep_wait();               // the partials come from the LM-head kernel
  // partial slots per row over the plan's launches (header word)
  const int slots = MODE == MERGE_GATHERED ? a.n_parts : a.n_rows[HDR_SLOTS];

  // ---- a3: merge of the partial slots
  {
    const int jj = threadIdx.x % LP;
    const int g = threadIdx.x / LP;
    float m = -INFINITY, s = 0.f;
    int arg = 0x7fffffff;
    // partial slots the workspace holds (index checks of the bounds-checked build)
    const int64_t part_n = MODE == MERGE_GATHERED
                               ? static_cast<int64_t>(a.n_parts) * a.P
                               : static_cast<int64_t>(plan_max_slots(a.plan)) * a.P;
    int r = -1;  // the slot index of this position: its compacted row, or (gathered) the position itself
    if (jj < L && index_ok(base + jj, a.P, a.status)) {
      if constexpr (MODE == MERGE_GATHERED)
        r = (a.pos_masked[base + jj] != 0 && (a.block_flags[blk] & 1u)) ? static_cast<int>(base + jj) : -1;
      else
        r = a.rowpos[base + jj];
    }
    if (g == 0) sm_live[jj] = r >= 0;
    if (r >= 0 && index_ok(r, a.P, a.status)) {
#pragma unroll 1
      for (int slot = g; slot < slots; slot += BATCH * GROUPS) {
        float pm[BATCH], ps[BATCH];
        int pa[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
          const int64_t o = static_cast<int64_t>(slot + u * GROUPS) * a.P + r;
          const bool in = slot + u * GROUPS < slots && index_ok(o, part_n, a.status);
          pm[u] = in ? a.part_m[o] : -INFINITY;
          ps[u] = in ? a.part_s[o] : 0.f;
          pa[u] = in ? a.part_a[o] : 0x7fffffff;
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) softmax_combine(m, s, arg, pm[u], ps[u], pa[u]);
      }
    }
    sm_m[jj][g] = m;
    sm_s[jj][g] = s;
    sm_a[jj][g] = arg;
  }
  __syncthreads();
  {
    // warp w: position w (LP = 32), or positions 2 w and 2 w + 1 in its half-warps (LP = 64)
    const int jj = (threadIdx.x / GROUPS), g = threadIdx.x % GROUPS;
    float m = sm_m[jj][g], s = sm_s[jj][g];
    int arg = sm_a[jj][g];
#pragma unroll
    for (int o = GROUPS / 2; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
      const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
      softmax_combine(m, s, arg, m2, s2, a2);
    }
    if (g == 0) {
      mg_m[jj] = m;
      mg_s[jj] = s;
      mg_a[jj] = arg;
    }
  }
  __syncthreads();
  if (warp != 0) return;

  if constexpr (MODE == MERGE_EMIT) {
    // one partial per window position, token ids of the whole vocabulary
#pragma unroll
    for (int h = 0; h < LP / 32; ++h) {
      const int jj = lane + 32 * h;
      if (jj < L) {
        float m = -INFINITY, s = 0.f;
        int arg = -1;
        if (sm_live[jj]) {
          m = mg_m[jj];
          s = mg_s[jj];
          arg = m == -INFINITY ? -1 : mg_a[jj] + a.vocab_offset;  // a shard holding only the mask token: nothing
        }
        a.emit_m[base + jj] = m;
        a.emit_s[base + jj] = s;
        a.emit_a[base + jj] = arg;
      }
    }
    return;
  }

  const uint32_t flags = a.block_flags[blk];
  const bool eligible = (flags & 2u) != 0;
  bool live[2] = {false, false};
  float conf[2] = {0.f, 0.f};
  int tok[2] = {-1, -1};
#pragma unroll
  for (int h = 0; h < LP / 32; ++h) {
    const int jj = lane + 32 * h;
    live[h] = jj < L && sm_live[jj];
    if (live[h]) {
      conf[h] = 1.f / mg_s[jj];  // the sum is >= 1: the maximum contributes exp(0)
      tok[h] = mg_a[jj];
    }
  }

  // fallback candidate: highest confidence among masked positions, lowest position on ties
  float best_c = -1.f;
  int best_j = 0x7fffffff;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int jj = lane + 32 * h;
    if (live[h] && (conf[h] > best_c || (conf[h] == best_c && jj < best_j))) {
      best_c = conf[h];
      best_j = jj;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float c2 = __shfl_xor_sync(0xffffffffu, best_c, o);
    const int j2 = __shfl_xor_sync(0xffffffffu, best_j, o);
    if (c2 > best_c || (c2 == best_c && j2 < best_j)) {
      best_c = c2;
      best_j = j2;
    }
  }
  const bool any_live = __any_sync(0xffffffffu, live[0] || live[1]);
  const bool take_fallback = eligible && any_live;

  const int seq = blk / a.n_slots;
  uint32_t bits[2] = {0u, 0u};
  for (int k = 0; k < a.taus.T; ++k) {
    const float tau = a.taus.tau[k];
    bool c0 = live[0] && conf[0] >= tau;
    bool c1 = live[1] && conf[1] >= tau;
    uint32_t b0 = __ballot_sync(0xffffffffu, c0);
    uint32_t b1 = __ballot_sync(0xffffffffu, c1);
    if ((b0 | b1) == 0u && take_fallback) {
      if (best_j < 32) {
        b0 = 1u << best_j;
        c0 = (lane == best_j);
      } else {
        b1 = 1u << (best_j - 32);
        c1 = (lane == best_j - 32);
      }
    }
    bits[0] |= static_cast<uint32_t>(c0) << k;
    bits[1] |= static_cast<uint32_t>(c1) << k;
    if (a.out_counts != nullptr && lane == 0) {
      const int cnt = __popc(b0) + __popc(b1);
      if (cnt) atomicAdd(a.out_counts + static_cast<int64_t>(seq) * a.taus.T + k, cnt);
    }
  }

#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int jj = lane + 32 * h;
    if (jj < L) {
      a.out_tokens[base + jj] = tok[h];
      a.out_conf[base + jj] = conf[h];
      a.out_commit[base + jj] = bits[h];
    }
  }
}

cudaError_t launch_merge_commit(const CommitArgs& a, cudaStream_t st, int mode) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.n_blocks, 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool wide = a.block_len > 32;
  switch (mode) {
    case MERGE_EMIT:
      return cudaLaunchKernelEx(&cfg, wide ? merge_commit_kernel<MERGE_EMIT, 64> : merge_commit_kernel<MERGE_EMIT, 32>, a);
    case MERGE_GATHERED:
      return cudaLaunchKernelEx(
          &cfg, wide ? merge_commit_kernel<MERGE_GATHERED, 64> : merge_commit_kernel<MERGE_GATHERED, 32>, a);
    default:
      return cudaLaunchKernelEx(&cfg, wide ? merge_commit_kernel<MERGE_ROWS, 64> : merge_commit_kernel<MERGE_ROWS, 32>, a);
  }
}

}  // namespace bd

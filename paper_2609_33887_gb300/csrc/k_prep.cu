// Preparation kernels of the commit step: compaction of the still-masked
// positions of active blocks, packing of their hidden rows, and the FP8 e4m3
// and NVFP4 -> bf16 weight decodes of the precision levers.
#include "checks.h"
#include "kernels.h"

namespace bd {

// ---------------------------------------------------------------------------
// Compaction and row packing in one launch. Only masked positions of active
// blocks need a prediction (App. F: the accept threshold resolves positions of
// active blocks). Rows keep ascending position order, so the masked positions
// of a block are consecutive rows.
//
// CTA 0 counts the live positions of the whole window, clears the per-sequence
// counts and writes the workspace header (N and the LM head's plan for N) with
// all its threads. CTA 1 + c owns positions [c * chunk, (c + 1) * chunk): it
// counts the live positions before its chunk itself (no inter-CTA
// communication), scans its chunk, writes idx / rowpos for it and packs the
// hidden rows of its live positions into hc (tensor-core paths), one warp per
// row with the whole row's loads in flight.
//
// Bound: latency on small windows, where the LM head waits for this kernel (an
// 8 x 2 x 32 bf16 window: the header 2.8 us and the rows 3.5 us after its
// start); HBM on large ones.
// Chunks are therefore as small as eight positions (a row per warp) until the
// grid has four CTAs per SM.
//
// The grid may be resident while the kernel before it still runs, and that
// kernel may write what this one reads (the sweep moves the window on in
// place): mask, flags and rows are read with plain loads behind griddep_wait,
// never through the read-only path (ld.global.nc holds only for memory that
// nobody writes during the kernel), and no pointer to them is __restrict__.
// ---------------------------------------------------------------------------
constexpr int PREP_THREADS = 256;
constexpr int PREP_WARPS = PREP_THREADS / 32;
constexpr int PREP_MAX_CHUNK = 2048;

__device__ __forceinline__ int live_at(const uint8_t* pos_masked, const uint8_t* block_flags, int p, int block_len) {
  return (pos_masked[p] != 0 && (block_flags[p / block_len] & 1u)) ? 1 : 0;
}

// This thread's share of the live positions in [0, n): 16 mask bytes per load
// where the array starts on a 16-byte boundary.
__device__ __forceinline__ int count_live(const uint8_t* pos_masked, const uint8_t* block_flags, int n,
                                          int block_len) {
  int cnt = 0;
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(pos_masked) & 15u) == 0) {
    const int nv = n / 16;
    const uint4* m4 = reinterpret_cast<const uint4*>(pos_masked);
    for (int v = threadIdx.x; v < nv; v += PREP_THREADS) {
      const uint4 q = m4[v];
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
      int b = 16 * v / block_len;
      int rem = 16 * v - b * block_len;  // position within block b
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (rem + 4 <= block_len) {  // the four positions lie in one block
          if (block_flags[b] & 1u) cnt += __popc(__vcmpne4(w[j], 0u)) >> 3;
          rem += 4;
          if (rem == block_len) {
            rem = 0;
            ++b;
          }
        } else {
          for (int i = 0; i < 4; ++i) {
            if (((w[j] >> (8 * i)) & 0xFFu) != 0 && (block_flags[b] & 1u)) ++cnt;
            if (++rem == block_len) {
              rem = 0;
              ++b;
            }
          }
        }
      }
    }
    done = nv * 16;
  }
  for (int p = done + threadIdx.x; p < n; p += PREP_THREADS) cnt += live_at(pos_masked, block_flags, p, block_len);
  return cnt;
}

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Two float32 values -> two E4M3 codes (round to nearest even, saturating at
// 448), `lo` in the low byte.
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}

// f16x2 bit pattern -> two float32 values (exact).
__device__ __forceinline__ float2 f16x2_bits_to_float2(uint32_t h2) {
  return __half22float2(*reinterpret_cast<const __half2*>(&h2));
}

__device__ __forceinline__ float2 bf16x2_bits_to_float2(uint32_t b2) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&b2));
}

__device__ __forceinline__ float amax8(const uint4& q) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
  float m = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 f = bf16x2_bits_to_float2(w[j]);
    m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
  }
  return m;
}

// One packed row in the making: `up` multiplies the elements, and eight
// (store8) or one (store1) of them are written in the format's codes.
template <int FMT>
struct RowOut {
  uint8_t* hi;  // the packed row (ROWS_E4M3X2: its hi terms)
  uint8_t* lo;  // ROWS_E4M3X2: its lo terms
  float up;

  __device__ __forceinline__ void store8(const uint4& q, int v) const {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    if constexpr (FMT == ROWS_F16_POW2) {
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 f = bf16x2_bits_to_float2(w[j]);
        const __half2 h2 = __floats2half2_rn(f.x * up, f.y * up);
        o[j] = *reinterpret_cast<const uint32_t*>(&h2);
      }
      reinterpret_cast<uint4*>(hi)[v] = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
      uint32_t oh[2] = {0u, 0u}, ol[2] = {0u, 0u};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 f = bf16x2_bits_to_float2(w[j]);
        const float y0 = __fmul_rn(f.x, up), y1 = __fmul_rn(f.y, up);
        const uint32_t h2 = f32x2_to_e4m3x2(y0, y1);
        oh[j >> 1] |= h2 << (16 * (j & 1));
        if constexpr (FMT == ROWS_E4M3X2) {
          const float2 back = f16x2_bits_to_float2(e4m3x2_to_f16x2(h2));
          ol[j >> 1] |= f32x2_to_e4m3x2(y0 - back.x, y1 - back.y) << (16 * (j & 1));
        }
      }
      reinterpret_cast<uint2*>(hi)[v] = make_uint2(oh[0], oh[1]);
      if constexpr (FMT == ROWS_E4M3X2) reinterpret_cast<uint2*>(lo)[v] = make_uint2(ol[0], ol[1]);
    }
  }

  __device__ __forceinline__ void store1(float x, int e) const {
    if constexpr (FMT == ROWS_F16_POW2) {
      reinterpret_cast<__half*>(hi)[e] = __float2half_rn(x * up);
    } else {
      const float y = __fmul_rn(x, up);
      const uint32_t h2 = f32x2_to_e4m3x2(y, 0.f);
      hi[e] = static_cast<uint8_t>(h2 & 0xFFu);
      if constexpr (FMT == ROWS_E4M3X2) {
        const float back = f16x2_bits_to_float2(e4m3x2_to_f16x2(h2)).x;
        lo[e] = static_cast<uint8_t>(f32x2_to_e4m3x2(y - back, 0.f) & 0xFFu);
      }
    }
  }
};

// The factor a row of largest magnitude amax is multiplied by before it is
// encoded, and the token scale that undoes it on the logits (0 for an all-zero row).
//
// ROWS_F16_POW2: 2^s with s = 15 - e for amax in [2^(e-1), 2^e), so the largest
// magnitude lands in [2^14, 2^15) and every bf16 value at or above 2^-14 after
// scaling is exact in f16; s at most 126 so 2^-s stays a normal float.
//
// ROWS_E4M3X2 (W8A16 on the 8-bit tensor path): 2^s with s = 134 - E for the
// biased exponent E of amax (the largest magnitude lands in [128, 256)),
// between -126 and 126 so 2^s and 2^-s stay normal floats. y = h * 2^s (exact)
// becomes hi = e4m3(y) and lo = e4m3(y - hi), both rounded to nearest even. y
// has at most 8 significant bits and y - hi (exact in float32) at most 4 more,
// so hi + lo == y exactly whenever |y| >= 2^-2, i.e. for every element of at
// least 2^-10 of the row's largest; a smaller element is off by at most 2^-10
// (half the smallest E4M3 step), 2^-17 of the row's largest.
//
// ROWS_E4M3 (W8A8): 448 / amax, code = e4m3(h * inv), scale = amax / 448; each
// float32 step is one correctly rounded operation.
template <int FMT>
__device__ __forceinline__ void row_factors(float amax, float* up, float* scale) {
  if constexpr (FMT == ROWS_E4M3) {
    *up = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
    *scale = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
  } else {
    const int E = static_cast<int>(__float_as_uint(amax) >> 23);
    // amax in [2^(E-127), 2^(E-126)) for E > 0; E = 0 (zero or below 2^-126) takes the cap
    const int sh = !(amax > 0.f) ? 0 : FMT == ROWS_F16_POW2 ? min(141 - E, 126) : max(min(134 - E, 126), -126);
    *up = __uint_as_float(static_cast<uint32_t>(sh + 127) << 23);  // 2^s, exact
    *scale = amax > 0.f ? __uint_as_float(static_cast<uint32_t>(127 - sh) << 23) : 0.f;
  }
}

// Bytes between packed rows: ldc counts 16-bit elements, or bytes for the 8-bit formats.
template <int FMT>
__device__ __forceinline__ int64_t packed_row_bytes(int64_t ldc) {
  return FMT == ROWS_BF16 || FMT == ROWS_F16_POW2 ? 2 * ldc : ldc;
}

// One warp packs the d elements of the bf16 row src into dst (16-byte aligned
// rows of row_bytes; ROWS_E4M3X2: the lo terms lo_offset bytes after the hi
// terms) and returns the row's token scale. Loads are issued ahead of the
// stores batch by batch: src and dst might alias for all the compiler knows.
template <int FMT, int RC>
__device__ __forceinline__ float pack_row(const __nv_bfloat16* src, int d, uint8_t* dst, int64_t lo_offset) {
  const int lane = threadIdx.x & 31, nvec = d / 8;
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  if constexpr (FMT == ROWS_BF16) {
    // 12 loads a lane: rows of up to 3072 elements in one batch (223 rows, d =
    // 2376, V = 35330: 54.9 us a step with 8, 54.3 with 12; with 16, 53.9, but
    // 4330 rows of d = 4296 lose 0.5%)
    constexpr int BATCH = 12;
    uint4* d4 = reinterpret_cast<uint4*>(dst);
    for (int v0 = lane; v0 < nvec; v0 += 32 * BATCH) {
      uint4 q[BATCH];
#pragma unroll
      for (int k = 0; k < BATCH; ++k)
        if (v0 + 32 * k < nvec) q[k] = s4[v0 + 32 * k];
#pragma unroll
      for (int k = 0; k < BATCH; ++k)
        if (v0 + 32 * k < nvec) d4[v0 + 32 * k] = q[k];
    }
    for (int e = nvec * 8 + lane; e < d; e += 32) reinterpret_cast<__nv_bfloat16*>(dst)[e] = src[e];
    return 1.f;
  } else {
    // rows of up to 32 * RC vectors are read once, into registers
    const bool cached = nvec <= 32 * RC;
    uint4 qc[RC];
    float amax = 0.f;
    if (cached) {
#pragma unroll
      for (int k = 0; k < RC; ++k) {
        const int v = lane + 32 * k;
        qc[k] = v < nvec ? s4[v] : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int k = 0; k < RC; ++k) amax = fmaxf(amax, amax8(qc[k]));
    } else {
#pragma unroll 4
      for (int v = lane; v < nvec; v += 32) amax = fmaxf(amax, amax8(s4[v]));
    }
    for (int e = nvec * 8 + lane; e < d; e += 32) amax = fmaxf(amax, fabsf(__bfloat162float(src[e])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    RowOut<FMT> out;
    float scale;
    row_factors<FMT>(amax, &out.up, &scale);
    out.hi = dst;
    out.lo = dst + lo_offset;
    if (cached) {
#pragma unroll
      for (int k = 0; k < RC; ++k) {
        const int v = lane + 32 * k;
        if (v < nvec) out.store8(qc[k], v);
      }
    } else {
      constexpr int BATCH = 4;
      for (int v0 = lane; v0 < nvec; v0 += 32 * BATCH) {
        uint4 q[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; ++k)
          if (v0 + 32 * k < nvec) q[k] = s4[v0 + 32 * k];
#pragma unroll
        for (int k = 0; k < BATCH; ++k)
          if (v0 + 32 * k < nvec) out.store8(q[k], v0 + 32 * k);
      }
    }
    for (int e = nvec * 8 + lane; e < d; e += 32) out.store1(__bfloat162float(src[e]), e);
    return scale;
  }
}

// FMT: the packed row format (ROWS_*). RC: vectors of a row a lane keeps in
// registers: 8 for rows of up to 2048 elements, else 20 (5120). The straight
// code for 20 costs a short row its instruction fetches: an 8 x 2 x 32 window's
// E4M3X2 rows (d = 2048) were packed 7.5 us after the kernel's start with it,
// 4.9 us without.
template <int FMT, int RC>
__global__ void __launch_bounds__(PREP_THREADS, 2) prep_rows_kernel(PrepArgs a) {
  __shared__ int red[2][PREP_WARPS];
  __shared__ int rows_s[PREP_MAX_CHUNK];
  __shared__ PlanScratch plan_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();  // every CTA of this grid is resident once all have got here
  griddep_wait();               // the caller's window, and the previous step's use of the workspace

  if (blockIdx.x == 0) {
    // the header's CTA
    const int cnt = warp_sum(count_live(a.pos_masked, a.block_flags, a.P, a.block_len));
    if (lane == 0) red[0][warp] = cnt;
    for (int i = tid; i < a.n_counts; i += PREP_THREADS) a.counts[i] = 0;
    __syncthreads();
    int n = 0;
#pragma unroll
    for (int w = 0; w < PREP_WARPS; ++w) n += red[0][w];
    plan_write_header(a.plan, n, a.n_rows, &plan_s);
    return;
  }

  const int p0 = (static_cast<int>(blockIdx.x) - 1) * a.chunk;
  const int p1 = min(a.P, p0 + a.chunk);
  // 1. live positions before this chunk, and the scan of the chunk, 256 positions at a time
  const int before = warp_sum(count_live(a.pos_masked, a.block_flags, p0, a.block_len));
  if (lane == 0) red[1][warp] = before;
  int prefix = 0, local_total = 0;
  for (int s0 = p0; s0 < p1; s0 += PREP_THREADS) {
    const int p = s0 + tid;
    const bool mine = p < p1 && live_at(a.pos_masked, a.block_flags, p, a.block_len);
    const uint32_t bal = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) red[0][warp] = __popc(bal);
    __syncthreads();
    if (s0 == p0) {
#pragma unroll
      for (int w = 0; w < PREP_WARPS; ++w) prefix += red[1][w];
    }
    int excl = local_total;
#pragma unroll
    for (int w = 0; w < PREP_WARPS; ++w) {
      const int c = red[0][w];
      if (w < warp) excl += c;
      local_total += c;
    }
    if (p < p1) {
      const int i = excl + __popc(bal & ((1u << lane) - 1u));
      if (mine) {
        if (index_ok(prefix + i, a.P, a.status)) a.idx[prefix + i] = p;
        rows_s[i] = p;
      }
      a.rowpos[p] = mine ? prefix + i : -1;
    }
    __syncthreads();
  }
  if (a.hidden == nullptr) return;

  // 2. pack the chunk's live rows
  const int64_t row_bytes = packed_row_bytes<FMT>(a.ldc);
  for (int i = warp; i < local_total; i += PREP_WARPS) {
    const int r = prefix + i;
    if (!index_ok(r, a.P, a.status)) continue;
    const float scale = pack_row<FMT, RC>(a.hidden + static_cast<int64_t>(rows_s[i]) * a.ld, a.d,
                                          static_cast<uint8_t*>(a.hc) + r * row_bytes, a.P * row_bytes);
    if (FMT != ROWS_BF16 && lane == 0) a.tok_scale[r] = scale;
  }
}

// Positions per packing CTA: four CTAs per SM, at least a row per warp.
int prep_chunk(int P, int sm_count) {
  int chunk = (P + 4 * sm_count - 1) / (4 * sm_count);
  chunk = (chunk + PREP_WARPS - 1) / PREP_WARPS * PREP_WARPS;
  return chunk > PREP_MAX_CHUNK ? PREP_MAX_CHUNK : chunk;
}

// Launched with programmatic stream serialisation behind the kernel before it
// (every CTA waits for that kernel first), except into a stream capture, whose
// first node may follow copies and other streams' work.
template <typename... Params, typename... Args>
static cudaError_t launch_behind(void (*kern)(Params...), int grid, cudaStream_t st, const Args&... args) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cs);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid), 1, 1);
  cfg.blockDim = dim3(PREP_THREADS, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

cudaError_t launch_prep_rows(const PrepArgs& args, int row_format, int sm_count, cudaStream_t st) {
  if (row_format != ROWS_BF16 && (args.tok_scale == nullptr || args.hc == nullptr)) return cudaErrorInvalidValue;
  PrepArgs a = args;
  a.chunk = prep_chunk(a.P, sm_count);
  const int grid = 1 + (a.P + a.chunk - 1) / a.chunk;
  const bool small = a.d <= 2048;
  auto* kern = row_format == ROWS_F16_POW2 ? (small ? prep_rows_kernel<ROWS_F16_POW2, 8> : prep_rows_kernel<ROWS_F16_POW2, 20>)
               : row_format == ROWS_E4M3   ? (small ? prep_rows_kernel<ROWS_E4M3, 8> : prep_rows_kernel<ROWS_E4M3, 20>)
               : row_format == ROWS_E4M3X2 ? (small ? prep_rows_kernel<ROWS_E4M3X2, 8> : prep_rows_kernel<ROWS_E4M3X2, 20>)
                                           : prep_rows_kernel<ROWS_BF16, 1>;
  return launch_behind(kern, grid, st, a);
}

// ---------------------------------------------------------------------------
// Verification rows need no compaction: every row is live, and the LM head
// reads the caller's rows in place. Row r = q * (n_draft + 1) + i verifies draft
// token i of request q (i < n_draft); the last row of a request verifies nothing.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(PREP_THREADS) prep_verify_kernel(PrepVerifyArgs a) {
  __shared__ PlanScratch plan_s;
  griddep_launch_dependents();
  griddep_wait();
  const int D = a.n_draft, R = a.n_req * (D + 1);
  if (blockIdx.x == 0) {  // N and the plan for it
    plan_write_header(a.plan, R, a.n_rows, &plan_s);
    return;
  }
  for (int r = (blockIdx.x - 1) * PREP_THREADS + threadIdx.x; r < R; r += (gridDim.x - 1) * PREP_THREADS) {
    const int q = r / (D + 1), i = r % (D + 1);
    a.idx[r] = r;
    a.draft_row[r] = i < D ? a.draft[q * D + i] : -1;
  }
}

cudaError_t launch_prep_verify(const PrepVerifyArgs& a, cudaStream_t st) {
  const int R = a.n_req * (a.n_draft + 1);
  int grid = (R + PREP_THREADS - 1) / PREP_THREADS;
  if (grid < 1) grid = 1;
  if (grid > 1024) grid = 1024;
  return launch_behind(prep_verify_kernel, 1 + grid, st, a);
}

// ---------------------------------------------------------------------------
// FP8 E4M3 -> bf16. Every e4m3 value (subnormals included) is exactly
// representable in f16 and in bf16, so the decode is exact; the per-row
// scale is applied later, to the fp32 logit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t e4m3x2_to_bf16x2(uint16_t two) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(two));
  __half2 h = *reinterpret_cast<__half2*>(&h2);
  float2 f = __half22float2(h);
  __nv_bfloat162 b = __floats2bfloat162_rn(f.x, f.y);
  return *reinterpret_cast<uint32_t*>(&b);
}

// One warp per row (grid-stride over rows). The row is cut into 8-element
// chunks; lane l takes chunks l, l + 32, ..., so every warp load reads 256
// contiguous code bytes and every warp store writes 512 contiguous output
// bytes; four chunks per lane are in flight at once. No index needs a division.
__global__ void __launch_bounds__(256) dequant_e4m3_kernel(const uint8_t* __restrict__ w, int64_t ldw, int V, int d,
                                                           __nv_bfloat16* __restrict__ out, int64_t ldo) {
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  const int nchunk = (d + 7) / 8;
  for (int v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < V; v += warps) {
    const uint8_t* src_row = w + static_cast<int64_t>(v) * ldw;
    __nv_bfloat16* dst_row = out + static_cast<int64_t>(v) * ldo;
    for (int c0 = lane; c0 < nchunk; c0 += 128) {
      uint2 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        // 8 codes at 8c: inside the row (ldw % 16 == 0 and ldw >= d)
        if (c < nchunk) q[u] = __ldg(reinterpret_cast<const uint2*>(src_row + 8 * c));
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        if (c >= nchunk) break;
        uint4 o;
        o.x = e4m3x2_to_bf16x2(static_cast<uint16_t>(q[u].x & 0xFFFFu));
        o.y = e4m3x2_to_bf16x2(static_cast<uint16_t>(q[u].x >> 16));
        o.z = e4m3x2_to_bf16x2(static_cast<uint16_t>(q[u].y & 0xFFFFu));
        o.w = e4m3x2_to_bf16x2(static_cast<uint16_t>(q[u].y >> 16));
        __nv_bfloat16* dst = dst_row + 8 * c;
        if (8 * c + 8 <= d) {
          *reinterpret_cast<uint4*>(dst) = o;  // ldo % 8 == 0: 16-byte aligned
        } else {
          const __nv_bfloat16* ov = reinterpret_cast<const __nv_bfloat16*>(&o);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (8 * c + j < d) dst[j] = ov[j];
        }
      }
    }
  }
}

cudaError_t launch_dequant_e4m3(const uint8_t* w, int64_t ldw, int V, int d, void* out, int64_t ldo, int sm_count,
                                cudaStream_t st) {
  int grid = sm_count * 8;
  dequant_e4m3_kernel<<<grid, 256, 0, st>>>(w, ldw, V, d, static_cast<__nv_bfloat16*>(out), ldo);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// NVFP4 -> bf16. An E2M1 code is 1 sign bit, 2 exponent bits (bias 1) and 1
// mantissa bit; its value (1 + m/2) * 2^(e-1), or m/2 for e = 0, is built
// directly as a binary32 bit pattern. Times the E4M3 block scale the product
// has at most 5 significant bits, so the bf16 result is exact; the per-row
// scale is applied later, to the fp32 logit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float e2m1_value(uint32_t c) {
  const uint32_t e = (c >> 1) & 3u, m = c & 1u;
  const uint32_t mag = e == 0 ? (m ? 0x3F000000u : 0u) : (((126u + e) << 23) | (m << 22));
  return __uint_as_float(mag | ((c & 8u) << 28));
}

__device__ __forceinline__ float e4m3_value(uint8_t c) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(static_cast<uint16_t>(c)));
  return __half2float(__ushort_as_half(static_cast<unsigned short>(h2 & 0xffffu)));
}

// One warp per row (grid-stride over rows). The row is cut into 8-element
// chunks (4 code bytes, 16 output bytes); lane l takes chunks l, l + 32, ...,
// so every warp load reads 128 contiguous code bytes and every warp store
// writes 512 contiguous output bytes; four chunks per lane are in flight at
// once. Chunk c uses block scale c / 2. No index needs a division.
__global__ void __launch_bounds__(256) dequant_nvfp4_kernel(const uint8_t* __restrict__ codes, int64_t ldw,
                                                            const uint8_t* __restrict__ bs, int64_t ldbs, int V,
                                                            int d, __nv_bfloat16* __restrict__ out, int64_t ldo) {
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  const int nchunk = (d + 7) / 8;
  for (int v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < V; v += warps) {
    const uint8_t* crow = codes + static_cast<int64_t>(v) * ldw;
    const uint8_t* brow = bs + static_cast<int64_t>(v) * ldbs;
    __nv_bfloat16* orow = out + static_cast<int64_t>(v) * ldo;
    for (int c0 = lane; c0 < nchunk; c0 += 128) {
      uint32_t q[4];
      uint8_t sb[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        // 4 code bytes at 4c: inside the row (ldw % 16 == 0 and ldw >= ceil(d / 2))
        if (c < nchunk) {
          q[u] = __ldg(reinterpret_cast<const uint32_t*>(crow + 4 * c));
          sb[u] = brow[c >> 1];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        if (c >= nchunk) break;
        const float sc = e4m3_value(sb[u]);
        uint32_t ow[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t byte = (q[u] >> (8 * j)) & 0xFFu;
          __nv_bfloat162 pr = __floats2bfloat162_rn(e2m1_value(byte & 0xFu) * sc, e2m1_value(byte >> 4) * sc);
          ow[j] = *reinterpret_cast<uint32_t*>(&pr);
        }
        __nv_bfloat16* dst = orow + 8 * c;
        if (8 * c + 8 <= d) {
          *reinterpret_cast<uint4*>(dst) = make_uint4(ow[0], ow[1], ow[2], ow[3]);  // ldo % 8 == 0
        } else {
          const __nv_bfloat16* ov = reinterpret_cast<const __nv_bfloat16*>(ow);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (8 * c + j < d) dst[j] = ov[j];
        }
      }
    }
  }
}

cudaError_t launch_dequant_nvfp4(const uint8_t* codes, int64_t ldw, const uint8_t* bs, int64_t ldbs, int V, int d,
                                 void* out, int64_t ldo, int sm_count, cudaStream_t st) {
  int grid = sm_count * 8;
  dequant_nvfp4_kernel<<<grid, 256, 0, st>>>(codes, ldw, bs, ldbs, V, d, static_cast<__nv_bfloat16*>(out), ldo);
  return cudaGetLastError();
}

}  // namespace bd

// LM-head projection + mask-suppressed softmax statistics with fp32 FMA on
// the CUDA cores. This is the exact-fp32 path (fp32 hidden states and head),
// and it accepts bf16 / e4m3 / NVFP4 heads too. Same band plan and partial
// layout as the tensor-core kernels. The verification instantiation (VERIFY =
// true) also carries the entropy accumulator and the logit of each row's
// draft entry.
//
// A CTA of 128 threads computes tiles of 8 R rows x 16 C vocabulary entries:
// a thread holds R x C logits (R <= 12 rows, C columns). R follows from the row
// count (simt_group_rows), so a 77-row window is one group of 80 rows.
// Both operands sit in shared memory as they are stored, 16 columns of d per
// stage in rows of 20 floats (an odd number of 16-byte units: eight rows read
// at one column hit different banks), filled by 16-byte asynchronous copies
// into a ring of stages that runs on across the tiles of a unit.
//
// C = 8 and 7 are bound by instruction issue on the SMs that hold most tiles
// (FMAs are 78% of the instructions, shared memory a third busy): 18 reads of
// four columns of d feed 320 products of a thread. 77 rows, d = 1024, V =
// 50304: 201 us with C = 7 (450 tiles on 152 SMs), 223 us with C = 8 (393 tiles,
// so the SMs with three of them set the time of all). With one column of eight
// rows per thread the same LM head took 520 us, bound by nine reads per eight
// products. C = 2 and 4 serve vocabularies that would leave most SMs without a
// wider tile, with more, smaller stages in flight (32 rows, d = 256, V = 4096:
// 17 us, latency). The host chooses C (simt_tile).
#include <atomic>
#include <cfloat>
#include <cuda_fp16.h>

#include "bdcommit.h"
#include "kernels.h"

namespace bd {

namespace {

constexpr int KC = 16;      // columns of d per stage
constexpr int KS = KC + 4;  // row stride of a stage
constexpr int THREADS = 128;
constexpr int MAX_R = 12;
// shared memory of an SM, and what the system keeps of it per CTA
constexpr size_t SMEM_PER_SM = 228 * 1024, SMEM_RESERVED = 1024;

template <int C>
__host__ __device__ constexpr int bn_of() { return 16 * C; }  // entries per tile
template <int C>
__host__ __device__ constexpr int stages_of() { return C > 4 ? 3 : C == 4 ? 4 : 6; }

__device__ __forceinline__ float load_h(const void* p, int64_t i, int dt) {
  if (dt == BD_F32) return static_cast<const float*>(p)[i];
  return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
}

// The smaller of two, NaN if either is.
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

__device__ __forceinline__ float e4m3_to_float(uint8_t c) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(static_cast<uint16_t>(c)));
  return __half2float(__ushort_as_half(static_cast<unsigned short>(h2 & 0xffffu)));
}

// Element k of head row v. NVFP4: the E2M1 nibble k (low nibble first) times
// the E4M3 scale of its 16-element block; the value is built from the code's
// bit fields (sign, 2-bit exponent with bias 1, 1-bit mantissa).
__device__ __forceinline__ float load_w(const SimtArgs& a, int v, int k) {
  const int64_t row = static_cast<int64_t>(v) * a.ldw;
  if (a.wdtype == BD_F32) return static_cast<const float*>(a.w)[row + k];
  if (a.wdtype == BD_BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(a.w)[row + k]);
  const uint8_t* p = static_cast<const uint8_t*>(a.w) + row;
  if (a.wdtype == BD_E4M3) return e4m3_to_float(p[k]);
  const uint8_t byte = p[k / 2];
  const uint32_t c = (k & 1) ? (byte >> 4) : (byte & 0xFu);
  const uint32_t e = (c >> 1) & 3u, m = c & 1u;
  const uint32_t mag = e == 0 ? (m ? 0x3F000000u : 0u) : (((126u + e) << 23) | (m << 22));
  return __uint_as_float(mag | ((c & 8u) << 28)) * e4m3_to_float(a.wbs[static_cast<int64_t>(v) * a.ldbs + k / 16]);
}

// Asynchronous copy of four floats to shared memory, of which the first n are
// read and the others zeroed (16-byte aligned addresses), and of one float.
__device__ __forceinline__ void copy16(float* dst, const float* src, int n) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(4 * n) : "memory");
}
__device__ __forceinline__ void copy4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int C>
struct Stage {
  float h[8 * MAX_R][KS];  // hidden rows
  float w[bn_of<C>()][KS];  // head rows
};

// How a stage's operands get to shared memory: as float vectors, as single
// floats (rows that do not start on 16-byte boundaries), or decoded.
enum : int { LOAD_VEC = 0, LOAD_FLOAT = 1, LOAD_DECODE = 2 };

template <int C, bool VERIFY>
struct SimtSmem {
  Stage<C> st[stages_of<C>()];
  // running softmax state of each thread's rows over its columns
  float m[MAX_R][THREADS], s[MAX_R][THREADS];
  int a[MAX_R][THREADS];
  float t[VERIFY ? MAX_R : 1][THREADS];
  int rix[8 * MAX_R];  // the m-tile's hidden rows (-1 past N)
  float rx[8 * MAX_R];  // VERIFY: the draft entry's logit of each row, and the entry
  int xd[8 * MAX_R];
};

// One unit: its m-tile's 8 R rows against v-tiles [vt0, vt_end). A thread's
// rows are tr + 8 i, its columns tc + 16 j.
template <int R, int C, bool VERIFY>
__device__ __forceinline__ void run_unit(const SimtArgs& a, SimtSmem<C, VERIFY>& sm, int vt0, int vt_end, int load) {
  constexpr int BN = bn_of<C>(), S = stages_of<C>();
  constexpr int ROWS = BN + 8 * R;  // staged rows: the head's, then the hidden ones
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tr = (warp >> 1) * 4 + (lane >> 3);
  const int tc = (warp & 1) * 8 + (lane & 7);
  const int nk = cdiv(a.d, KC);
  const int total = (vt_end - vt0) * nk;

  int ivt = vt0, ik = 0, islot = 0;  // the next step to load: v-tile, first column, stage
  auto issue = [&]() {
    Stage<C>& st = sm.st[islot];
    if (load == LOAD_VEC) {
      const int c = tid & 3, k = ik + 4 * c;  // this thread's vector of every 32nd row
      const int n = min(4, a.d - k);          // floats of it that exist
#pragma unroll
      for (int p = 0; p < (ROWS + 31) / 32; ++p) {
        const int r = (tid >> 2) + 32 * p;
        if (32 * p + 32 <= BN || r < BN) {
          const int v = ivt * BN + r;
          const bool in = v < a.V && n > 0;
          copy16(&st.w[r][4 * c], static_cast<const float*>(a.w) + (in ? static_cast<int64_t>(v) * a.ldw + k : 0),
                 in ? n : 0);
        } else if (r < ROWS) {
          const int src = sm.rix[r - BN];
          const bool in = src >= 0 && n > 0;
          copy16(&st.h[r - BN][4 * c],
                 static_cast<const float*>(a.hidden) + (in ? static_cast<int64_t>(src) * a.ldh + k : 0), in ? n : 0);
        }
      }
    } else {
      const int k = ik + (tid & 15);
#pragma unroll 4
      for (int r = tid >> 4; r < ROWS; r += THREADS / 16) {
        const bool head = r < BN;
        const int row = head ? ivt * BN + r : sm.rix[r - BN];
        const bool in = k < a.d && (head ? row < a.V : row >= 0);
        float* dst = head ? &st.w[r][tid & 15] : &st.h[r - BN][tid & 15];
        if (load == LOAD_FLOAT) {
          const float* base = static_cast<const float*>(head ? a.w : a.hidden);
          copy4(dst, base + (in ? static_cast<int64_t>(row) * (head ? a.ldw : a.ldh) + k : 0), in);
        } else {
          *dst = !in ? 0.f : head ? load_w(a, row, k) : load_h(a.hidden, static_cast<int64_t>(row) * a.ldh + k, a.hdtype);
        }
      }
    }
    if (++islot == S) islot = 0;
    ik += KC;
    if (ik >= a.d) {
      ik = 0;
      ++ivt;
    }
  };

#pragma unroll 1
  for (int i = 0; i < S - 1; ++i) {
    if (i < total) issue();
    copy_commit();
  }
  int slot = 0, step = 0;
#pragma unroll 1
  for (int vt = vt0; vt < vt_end; ++vt) {
    float acc[R][C];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < C; ++j) acc[i][j] = 0.f;
#pragma unroll 1
    for (int kb = 0; kb < nk; ++kb, ++step) {
      copy_wait<S - 2>();
      __syncthreads();  // this step has landed for every thread, and the stage loaded next has been read by all
      if (step + S - 1 < total) issue();
      copy_commit();
      const Stage<C>& st = sm.st[slot];
#pragma unroll 1
      for (int k = 0; k < KC; k += 4) {
        float4 w[C];
#pragma unroll
        for (int j = 0; j < C; ++j) w[j] = *reinterpret_cast<const float4*>(&st.w[tc + 16 * j][k]);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float4 h = *reinterpret_cast<const float4*>(&st.h[tr + 8 * i][k]);
#pragma unroll
          for (int j = 0; j < C; ++j) {
            acc[i][j] = fmaf(h.x, w[j].x, acc[i][j]);
            acc[i][j] = fmaf(h.y, w[j].y, acc[i][j]);
            acc[i][j] = fmaf(h.z, w[j].z, acc[i][j]);
            acc[i][j] = fmaf(h.w, w[j].w, acc[i][j]);
          }
        }
      }
      if (++slot == S) slot = 0;
    }
    // the tile's logits into each row's running state over this thread's columns
    int col[C];
    float sc[C];
    bool dead[C];
#pragma unroll
    for (int j = 0; j < C; ++j) {
      col[j] = vt * BN + 16 * j + tc;
      dead[j] = col[j] >= a.V || col[j] == a.mask_id;
      sc[j] = a.wscale != nullptr && col[j] < a.V ? a.wscale[col[j]] : 1.f;
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      float x[C];
      float cm = -INFINITY;
#pragma unroll
      for (int j = 0; j < C; ++j) {
        x[j] = dead[j] ? -INFINITY : acc[i][j] * sc[j];
        cm = fmaxf(cm, x[j]);
      }
      if constexpr (VERIFY) {
        const int d_at = sm.xd[tr + 8 * i];
#pragma unroll
        for (int j = 0; j < C; ++j)
          if (col[j] == d_at && !dead[j]) sm.rx[tr + 8 * i] = x[j];  // one thread of the CTA holds the draft entry
      }
      float m = sm.m[i][tid], s = sm.s[i][tid], t = VERIFY ? sm.t[VERIFY ? i : 0][tid] : 0.f;
      if (cm > m) {
        int arg = 0;
#pragma unroll
        for (int j = C - 1; j >= 0; --j)
          if (x[j] == cm) arg = col[j];
        sm.a[i][tid] = arg;
        if (m != -INFINITY) {
          const float dm = (m - cm) * LOG2E;
          const float f = ex2_approx(dm);
          if constexpr (VERIFY) t = f * fmaf(dm, s, t);
          s *= f;
        }
        m = cm;
      }
      if (m != -INFINITY) {
        // an infinite maximum (logits that overflowed) counts 1 like any other:
        // u is cut at 0, against the largest finite number; NaN stays NaN
        const float base = fminf(m, FLT_MAX);
#pragma unroll
        for (int j = 0; j < C; ++j) {
          const float u = min_nan((x[j] - base) * LOG2E, 0.f);
          const float e = ex2_approx(u);
          s += e;
          // -inf logits give e = 0; clamping u keeps e * u at 0
          if constexpr (VERIFY) t = fmaf(e, fmaxf(u, -256.f), t);
        }
      }
      sm.m[i][tid] = m;
      sm.s[i][tid] = s;
      if constexpr (VERIFY) sm.t[VERIFY ? i : 0][tid] = t;
    }
  }
  copy_wait<0>();
}

}  // namespace

template <int C, bool VERIFY>
__global__ void __launch_bounds__(THREADS, simt_ctas(bn_of<C>(), VERIFY)) lmhead_simt_kernel(SimtArgs a) {
  static_assert(simt_ctas(bn_of<C>(), VERIFY) * (sizeof(SimtSmem<C, VERIFY>) + SMEM_RESERVED) <= SMEM_PER_SM,
                "the CTAs the plan counts on fit an SM");
  extern __shared__ __align__(16) uint8_t smem_raw[];
  SimtSmem<C, VERIFY>& sm = *reinterpret_cast<SimtSmem<C, VERIFY>*>(smem_raw);
  const int tid = threadIdx.x;
  griddep_wait();  // idx and N come from the preceding kernel
  const int n_rows = a.n_rows[HDR_N];
  const int rows = plan_bm(a.plan, n_rows);  // 8 R
  const bool f32 = a.wdtype == BD_F32 && a.hdtype == BD_F32;
  const bool vec = ((reinterpret_cast<uintptr_t>(a.w) | reinterpret_cast<uintptr_t>(a.hidden)) & 15u) == 0 &&
                   ((a.ldw | a.ldh) & 3) == 0;
  const int load = !f32 ? LOAD_DECODE : vec ? LOAD_VEC : LOAD_FLOAT;

  TileIter it;
  it.init(a.plan, a.n_rows);
  while (it.next_unit()) {
    const int r0 = it.m_tile * rows;
    static_assert(8 * MAX_R <= THREADS, "a thread per row");
    if (tid < 8 * MAX_R) {
      sm.rix[tid] = tid < rows && r0 + tid < n_rows ? a.idx[r0 + tid] : -1;
      if constexpr (VERIFY) {
        sm.rx[tid] = -INFINITY;
        sm.xd[tid] = tid < rows && r0 + tid < n_rows ? a.draft_row[r0 + tid] : -1;
      }
    }
#pragma unroll
    for (int i = 0; i < MAX_R; ++i) {
      sm.m[i][tid] = -INFINITY;
      sm.s[i][tid] = 0.f;
      sm.a[i][tid] = 0x7fffffff;
      if constexpr (VERIFY) sm.t[VERIFY ? i : 0][tid] = 0.f;
    }
    __syncthreads();
    switch (rows / 8) {
      case 1: run_unit<1, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 2: run_unit<2, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 3: run_unit<3, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 4: run_unit<4, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 5: run_unit<5, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 6: run_unit<6, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 7: run_unit<7, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 8: run_unit<8, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      case 10: run_unit<10, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
      default: run_unit<12, C, VERIFY>(a, sm, it.vt, it.vt_end, load); break;
    }
    __syncthreads();
    // row r's states: the 16 threads that hold its columns
    if (tid < rows && r0 + tid < n_rows) {
      const int tr = tid & 7, i = tid >> 3;
      float M = -INFINITY, S = 0.f, T = 0.f;
      int A = 0x7fffffff;
#pragma unroll 4
      for (int tc = 0; tc < 16; ++tc) {
        const int src = ((tr >> 2) * 2 + (tc >> 3)) * 32 + (tr & 3) * 8 + (tc & 7);
        if constexpr (VERIFY)
          softmax_combine_t(M, S, A, T, sm.m[i][src], sm.s[i][src], sm.a[i][src], sm.t[VERIFY ? i : 0][src]);
        else
          softmax_combine(M, S, A, sm.m[i][src], sm.s[i][src], sm.a[i][src]);
      }
      const int64_t o = static_cast<int64_t>(it.part) * a.P + r0 + tid;
      a.part_m[o] = M;
      a.part_s[o] = S;
      a.part_a[o] = A;
      if constexpr (VERIFY) {
        a.part_t[o] = T;
        a.part_x[o] = sm.rx[tid];
      }
    }
    __syncthreads();
  }
  griddep_launch_dependents();
}

template <int C, bool VERIFY>
static cudaError_t launch_simt(const SimtArgs& a, cudaStream_t st) {
  // the shared-memory opt-in is set once per device (not again inside a graph capture)
  static std::atomic<uint64_t> opted_in{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if ((opted_in.load() & bit) == 0) {
    e = cudaFuncSetAttribute(lmhead_simt_kernel<C, VERIFY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(SimtSmem<C, VERIFY>)));
    if (e != cudaSuccess) return e;
    opted_in.fetch_or(bit);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.plan.G, 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = sizeof(SimtSmem<C, VERIFY>);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lmhead_simt_kernel<C, VERIFY>, a);
}

cudaError_t launch_lmhead_simt(const SimtArgs& a, cudaStream_t st) {
  const bool verify = a.part_t != nullptr;
  switch (a.plan.BN) {
    case bn_of<2>(): return verify ? launch_simt<2, true>(a, st) : launch_simt<2, false>(a, st);
    case bn_of<4>(): return verify ? cudaErrorInvalidValue : launch_simt<4, false>(a, st);
    case bn_of<7>(): return verify ? launch_simt<7, true>(a, st) : launch_simt<7, false>(a, st);
    case bn_of<8>(): return verify ? launch_simt<8, true>(a, st) : launch_simt<8, false>(a, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace bd

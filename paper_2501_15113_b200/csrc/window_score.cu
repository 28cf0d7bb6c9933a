// Observation-window scores (Eq. 12, Eq. 13): for every unit
//   S = Q_win K^T / sqrt(d), causal mask on the last L keys, row softmax,
//   C[j] = mean over the unit's G*L window rows of the normalised weights.
//
// Two-pass path on the CUDA cores for fp32 inputs with up to 32 window rows; the others run on the tensor cores, where splitting
// the keys into planes costs the same whatever the rows.  Both passes here and there: 128 units of 3000 keys, d = 128, 16 rows 189
// and 189 us, 24 rows 281 and 191, 32 rows 286 and 193; 32 units of 6001 keys, d = 64, 24 and 32 rows 90 and 83, 64 rows 150 and
// 83, 128 rows 250 and 93.  So the kernels are level at 16 rows, and the line at 32 is higher than these figures put it:
//   pass 1  per (unit, 256-key chunk): row maxima and exp-sums  -> partial stats
//   reduce  per unit: combine chunks -> (row max, 1 / row sum); units of up to 32 chunks need no launch for it,
//           their pass-2 blocks combine the chunks themselves
//   pass 2  per (unit, chunk): recompute S, C[j] = sum_i exp(s_ij - max_i) / Z_i / rows
// Scores are kept in log2 units (scaled by log2(e)/sqrt(d)) so exp is one ex2.
//
// Bound by the fp32 FMA rate (2 * rows * d flop per key and pass), so each pass is a register-tiled product: a thread
// holds KPT keys x RPT rows, fed by 16-byte shared-memory reads along d, and keeps its own running (max, sum) per row, so
// that lanes meet once per chunk instead of twice per row and tile.
#include "common.cuh"

namespace taskkv {

namespace {

constexpr int kTile = 128;      // keys per tile
constexpr int kBlock = 256;     // threads
constexpr int kDepth = 64;      // elements of d staged in shared memory at a time
constexpr int kPitch = kDepth + 4;   // floats per staged key row: 16-byte reads of consecutive rows hit all banks
constexpr int kFoldChunks = 32; // units of up to this many chunks are folded by the pass-2 blocks

// How a block's 256 threads cover 128 keys x ROWS window rows.
template <int ROWS>
struct WinTile {
  static constexpr int RPT = 4;
  static constexpr int NTY = ROWS / RPT;
  static constexpr int NTX = kBlock / NTY;
  static constexpr int KPT = kTile / NTX;
  static constexpr int PARTS = kBlock / ROWS;    // threads that share a row's fold over the chunks
};

template <int D, int ROWS>
constexpr size_t win_smem() {
  return ((size_t)ROWS * (D + 4) + (size_t)kTile * kPitch + 2 * (size_t)ROWS) * sizeof(float);
}

// (max, sum) pairs in log2 units: a <- a + b.
__device__ __forceinline__ void fold_pair(float2& a, const float2 b) {
  if (b.x > -INFINITY) {
    const float M = fmaxf(a.x, b.x);
    a.y = a.y * exp2f(a.x - M) + b.y * exp2f(b.x - M);
    a.x = M;
  }
}

// (row max, 1 / row sum) of every row of unit u from its chunks' partials, by the whole block, into out[ROWS] (shared
// memory); tmp: kBlock pairs.  The order is fixed by the unit's own length.
template <int ROWS>
__device__ void fold_unit(const DeviceProblem& p, int u, int chunks, float2* tmp, float2* out) {
  constexpr int PARTS = WinTile<ROWS>::PARTS;
  const int row = threadIdx.x % ROWS, part = threadIdx.x / ROWS;
  const float2* src = reinterpret_cast<const float2*>(p.stat_part) + (size_t)u * p.chunks_max * p.rows_pad + row;
  float2 a = make_float2(-INFINITY, 0.f);
  if (row < p.rows) {
    for (int c = part; c < chunks; c += 4 * PARTS) {
      float2 o[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        o[i] = c + i * PARTS < chunks ? src[(size_t)(c + i * PARTS) * p.rows_pad] : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int i = 0; i < 4; ++i) fold_pair(a, o[i]);
    }
  }
  tmp[threadIdx.x] = a;
  __syncthreads();
  if (part == 0) {
#pragma unroll
    for (int q = 1; q < PARTS; ++q) fold_pair(a, tmp[q * ROWS + row]);
    out[row] = (row < p.rows && a.y > 0.f) ? make_float2(a.x, 1.0f / a.y) : make_float2(0.f, 0.f);
  }
  __syncthreads();
}

// fold: pass 2 combines the chunks itself (p.stat is not used).
template <int D, int ROWS, int PASS>
__global__ void __launch_bounds__(kBlock) window_pass_kernel(DeviceProblem p, UnitRange ur, int grid_chunks, int fold) {
  using W = WinTile<ROWS>;
  constexpr int RPT = W::RPT, NTY = W::NTY, NTX = W::NTX, KPT = W::KPT;
  using T = float;
  constexpr int VN = Vec16<T>::N;
  constexpr int VPR = kDepth / VN;                       // 16-byte vectors of one key row of a stage
  constexpr int VPT = kTile * VPR / kBlock;              // vectors per thread and stage
  constexpr int QP = D + 4;
  extern __shared__ __align__(16) float win_mem[];
  float* Qs = win_mem;                                                  // [ROWS][D + 4]
  float* Ks = Qs + ROWS * QP;                                           // [kTile][kPitch]; later scratch
  float2* st = reinterpret_cast<float2*>(Ks + kTile * kPitch);          // [ROWS]  pass 2: (max, 1 / sum)

  const int u = ur.unit(blockIdx.x / grid_chunks);
  const int chunk = blockIdx.x % grid_chunks;
  const int N = p.unit_N[u];
  const int key0 = chunk * kScoreChunk;
  if (key0 >= N) return;
  const int key_end = min(N, key0 + kScoreChunk);
  const int L = p.L;
  const int tid = threadIdx.x, tx = tid % NTX, ty = tid / NTX;

  // a stage is kDepth elements of 128 key rows; its global loads are issued before the stage before it is used
  const unsigned char* kbase = static_cast<const unsigned char*>(p.k_ptr[u]);
  const int stages = (key_end - key0 + kTile - 1) / kTile * (D / kDepth);
  uint4 pre[VPT];
  auto fetch = [&](int s) {
    const int t0 = key0 + s / (D / kDepth) * kTile, d0 = s % (D / kDepth) * kDepth;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int v = tid + i * kBlock, r = v / VPR, c = v % VPR;
      pre[i] = t0 + r < N ? *reinterpret_cast<const uint4*>(kbase + ((size_t)(t0 + r) * D + d0) * sizeof(T) + (size_t)c * 16)
                          : make_uint4(0, 0, 0, 0);
    }
  };
  fetch(0);
  // Q rows of the unit's G heads: [rows][d] contiguous, converted to fp32 once
  const uint4* q = static_cast<const uint4*>(p.q_ptr[u]);
  for (int v = tid; v < ROWS * (D / VN); v += kBlock) {
    const int r = v / (D / VN), c = v % (D / VN);
    float f[VN];
    Vec16<T>::unpack(r < p.rows ? q[v] : make_uint4(0, 0, 0, 0), f);
#pragma unroll
    for (int h = 0; h < VN; h += 4) *reinterpret_cast<float4*>(Qs + r * QP + c * VN + h) = make_float4(f[h], f[h + 1], f[h + 2], f[h + 3]);
  }
  if (PASS == 2) {
    grid_dependency_wait();                              // the statistics come from the launch before
    if (fold) {
      fold_unit<ROWS>(p, u, (N + kScoreChunk - 1) / kScoreChunk, reinterpret_cast<float2*>(Ks), st);
    } else {
      for (int i = tid; i < ROWS; i += kBlock)
        st[i] = i < p.rows ? reinterpret_cast<const float2*>(p.stat)[(size_t)u * p.rows_pad + i] : make_float2(0.f, 0.f);
    }
  }

  const float scale2 = kLog2e * rsqrtf((float)D);
  // last key the thread's rows may see: window row (row % L) sits at position N - L + (row % L)
  int pos[RPT];
  float m[RPT], z[RPT];                                  // pass 1: running max and sum; pass 2: the row's pair
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int row = ty + NTY * j;
    pos[j] = row < p.rows ? N - L + row % L : -1;
    m[j] = -INFINITY;
    z[j] = 0.f;
  }
  float acc[KPT][RPT];
  for (int s = 0; s < stages; ++s) {
    __syncthreads();                                     // the previous stage's readers (and the fold) are done
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int v = tid + i * kBlock, r = v / VPR, c = v % VPR;
      float f[VN];
      Vec16<T>::unpack(pre[i], f);
#pragma unroll
      for (int h = 0; h < VN; h += 4) *reinterpret_cast<float4*>(Ks + r * kPitch + c * VN + h) = make_float4(f[h], f[h + 1], f[h + 2], f[h + 3]);
    }
    if (s + 1 < stages) fetch(s + 1);
    __syncthreads();
    const int t0 = key0 + s / (D / kDepth) * kTile, d0 = s % (D / kDepth) * kDepth;
    if (d0 == 0) {
#pragma unroll
      for (int i = 0; i < KPT; ++i)
#pragma unroll
        for (int j = 0; j < RPT; ++j) acc[i][j] = 0.f;
    }
#pragma unroll 2
    for (int dd = 0; dd < kDepth; dd += 4) {
      float4 kf[KPT];
#pragma unroll
      for (int i = 0; i < KPT; ++i) kf[i] = *reinterpret_cast<const float4*>(Ks + (tx + NTX * i) * kPitch + dd);
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const float4 qv = *reinterpret_cast<const float4*>(Qs + (ty + NTY * j) * QP + d0 + dd);
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
          acc[i][j] = fmaf(qv.x, kf[i].x, acc[i][j]);
          acc[i][j] = fmaf(qv.y, kf[i].y, acc[i][j]);
          acc[i][j] = fmaf(qv.z, kf[i].z, acc[i][j]);
          acc[i][j] = fmaf(qv.w, kf[i].w, acc[i][j]);
        }
      }
    }
    if (d0 + kDepth < D) continue;                       // (D = 128) the other half of the products comes next
    if (PASS == 1) {
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        float x[KPT], mt = -INFINITY;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
          x[i] = t0 + tx + NTX * i <= pos[j] ? acc[i][j] * scale2 : -INFINITY;
          mt = fmaxf(mt, x[i]);
        }
        if (mt > m[j]) {
          z[j] *= exp2f(m[j] - mt);
          m[j] = mt;
        }
        if (m[j] > -INFINITY) {
#pragma unroll
          for (int i = 0; i < KPT; ++i) z[j] += exp2f(x[i] - m[j]);
        }
      }
    } else {
      float cs[KPT];
#pragma unroll
      for (int i = 0; i < KPT; ++i) cs[i] = 0.f;
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const float2 ms = st[ty + NTY * j];
#pragma unroll
        for (int i = 0; i < KPT; ++i)
          if (t0 + tx + NTX * i <= pos[j]) cs[i] += exp2f(acc[i][j] * scale2 - ms.x) * ms.y;
      }
      __syncthreads();                                   // every thread is done with this tile's keys
#pragma unroll
      for (int i = 0; i < KPT; ++i) Ks[ty * kTile + tx + NTX * i] = cs[i];
      __syncthreads();
      if (tid < kTile && t0 + tid < N) {
        float c = 0.f;
#pragma unroll
        for (int y = 0; y < NTY; ++y) c += Ks[y * kTile + tid];
        p.C[p.c_off[u] + t0 + tid] = c * (1.0f / (float)p.rows);
      }
    }
  }

  if (PASS == 1) {
    grid_launch_dependents();
    __syncthreads();
    float2* red = reinterpret_cast<float2*>(Ks);         // [ROWS][NTX + 1]
#pragma unroll
    for (int j = 0; j < RPT; ++j) red[(ty + NTY * j) * (NTX + 1) + tx] = make_float2(m[j], z[j]);
    __syncthreads();
    if (tid < p.rows) {
      float2 a = make_float2(-INFINITY, 0.f);
      for (int x = 0; x < NTX; ++x) fold_pair(a, red[tid * (NTX + 1) + x]);
      reinterpret_cast<float2*>(p.stat_part)[((size_t)u * p.chunks_max + chunk) * p.rows_pad + tid] = a;
    }
  }
}

// The fold as a launch of its own, for units of many chunks: every pass-2 block would read all of them again.
template <int ROWS>
__global__ void __launch_bounds__(kBlock) window_reduce_kernel(DeviceProblem p, UnitRange ur) {
  __shared__ float2 tmp[kBlock], out[ROWS];
  const int u = ur.unit(blockIdx.x);
  grid_dependency_wait();
  grid_launch_dependents();
  fold_unit<ROWS>(p, u, (p.unit_N[u] + kScoreChunk - 1) / kScoreChunk, tmp, out);
  for (int i = threadIdx.x; i < p.rows; i += kBlock) reinterpret_cast<float2*>(p.stat)[(size_t)u * p.rows_pad + i] = out[i];
}

// Caller-supplied normalisers lse_i = ln sum_j exp(s_ij) of the window rows, in place of pass 1.  A unit's G*L rows
// are contiguous in [R][n][L].
__global__ void lse_to_stat_kernel(DeviceProblem p, int u0, const float* __restrict__ lse, LseFormat format) {
  const int lu = blockIdx.x, row = threadIdx.x;
  if (row >= p.rows) return;
  const float v = lse[(size_t)lu * p.rows + row] * kLog2e;
  float* st = p.stat + (size_t)(u0 + lu) * (2 * p.rows_pad);
  if (format == LSE_PAIR) {
    st[row] = v;
    st[p.rows_pad + row] = 1.0f / (float)p.rows;
  } else if (format == LSE_OFFSET) {
    st[row] = v + log2f((float)p.rows);
  } else {
    reinterpret_cast<float2*>(st)[row] = make_float2(v, 1.0f);
  }
}

template <int D, int ROWS>
cudaError_t launch_generic_rows(const DeviceProblem& p, int max_N, const WindowHostInfo& h, cudaStream_t s, int layer0,
                                int n_layers) {
  constexpr size_t smem = win_smem<D, ROWS>();
  static_assert((size_t)kTile * kPitch >= 2 * (size_t)ROWS * (WinTile<ROWS>::NTX + 1), "pass 1's pairs reuse the key tile");
  cudaError_t e;
  e = cudaFuncSetAttribute(window_pass_kernel<D, ROWS, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(window_pass_kernel<D, ROWS, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const UnitRange ur = layer_range(p, h.batch, layer0, n_layers);
  const int chunks = (max_N + kScoreChunk - 1) / kScoreChunk;
  const int64_t grid = (int64_t)chunks * ur.blocks;
  if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
  const int fold = !h.lse && chunks <= kFoldChunks ? 1 : 0;
  if (h.lse) {
    const int per_seq = p.R * p.n_kv;
    const size_t lse_skip = (size_t)(layer0 - h.base_layer) * p.n_heads * p.L;
    for (int b = 0; b < h.batch; ++b) {
      e = launch_lse_to_stat(p, b * per_seq + ur.first, ur.count, static_cast<const float*>(h.lse[b]) + lse_skip, LSE_CUDA_CORES, s);
      if (e != cudaSuccess) return e;
    }
  } else {
    {
      LaunchScope ls(K_WINDOW_STATS, s);
      window_pass_kernel<D, ROWS, 1><<<(unsigned)grid, kBlock, smem, s>>>(p, ur, chunks, 0);
    }
    if (!fold) {
      LaunchScope ls(K_WINDOW_REDUCE, s);
      e = launch_dependent(window_reduce_kernel<ROWS>, (unsigned)ur.blocks, kBlock, s, p, ur);
      if (e != cudaSuccess) return e;
    }
  }
  {
    LaunchScope ls(K_WINDOW_SCORES, s);
    if (h.lse) window_pass_kernel<D, ROWS, 2><<<(unsigned)grid, kBlock, smem, s>>>(p, ur, chunks, 0);
    else e = launch_dependent_smem(window_pass_kernel<D, ROWS, 2>, (unsigned)grid, kBlock, smem, s, p, ur, chunks, fold);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_generic(const DeviceProblem& p, int max_N, const WindowHostInfo& h, cudaStream_t s, int layer0,
                           int n_layers) {
  if (p.rows <= 16) return launch_generic_rows<D, 16>(p, max_N, h, s, layer0, n_layers);
  return launch_generic_rows<D, 32>(p, max_N, h, s, layer0, n_layers);
}

}  // namespace

cudaError_t launch_lse_to_stat(const DeviceProblem& p, int u0, int n_units, const float* lse, LseFormat format, cudaStream_t s) {
  LaunchScope ls(K_WINDOW_REDUCE, s);
  lse_to_stat_kernel<<<n_units, 128, 0, s>>>(p, u0, lse, format);
  return cudaGetLastError();
}

cudaError_t launch_window_scores(const DeviceProblem& p, int dtype, int max_N, const WindowHostInfo& h,
                                 cudaStream_t s, int layer0, int n_layers) {
  if (n_layers < 0) { layer0 = 0; n_layers = p.R; }
  if ((dtype == TASKKV_F32 && p.rows > 32) || window_tc_supported(p, dtype))
    return launch_window_scores_tc(p, dtype, h, s, layer0, n_layers);
  if (dtype != TASKKV_F32) return cudaErrorNotSupported;      // bf16 without the driver's tensor maps
  return p.d == 64 ? launch_generic<64>(p, max_N, h, s, layer0, n_layers) : launch_generic<128>(p, max_N, h, s, layer0, n_layers);
}

}  // namespace taskkv

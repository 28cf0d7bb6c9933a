// The exact semantic vector of Sec. III-A (Eq. 1-2): v = (sum_i A[i,:] / N) V with the full N x N causal attention
// matrix A of a head -- the quantity that the observation window (Eq. 12-15) approximates.  Quadratic in N: an
// analysis routine (how far is v' from v, do the two rank the heads alike), not part of the compression path.
//
// The N query rows of a head are cut into blocks of 128; block b sees the first 128 (b + 1) keys, and prefix_score_tc.cu
// gives its column sums C_b[j] = (1/128) sum_{i in block b} A[i, j].  Then
//   C[j] = 128 / (G N) * sum over the G query heads of the KV head, and over the blocks b >= j / 128, of C_b[j]
//   v    = sum_j C[j] V[j, :]
// with fixed summation orders.  K of a head (N d 2 bytes) is walked twice per block and stays in L2 meanwhile.
#include <algorithm>

#include "common.cuh"

namespace taskkv {

namespace {

constexpr int kBlockRows = 128;        // query rows per prefix window
constexpr int kSliceKeys = 512;        // keys per partial sum of v

// offset of block b's scores inside a head's area: blocks 0 .. b-1 hold 128, 256, ... floats
__host__ __device__ inline int64_t block_off(int64_t b) { return 64 * b * (b + 1); }

// One thread per key j of a KV head: the blocks' scores added in ascending (query head, block) order.
__global__ void __launch_bounds__(256) exact_colsum_kernel(const float* __restrict__ Cb, int nb, int G, int N,
                                                           float* __restrict__ c_full) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int kvh = blockIdx.y;
  if (j >= N) return;
  float s = 0.f;
  for (int g = 0; g < G; ++g) {
    const float* head = Cb + (int64_t)(kvh * G + g) * block_off(nb);
    for (int b = j / kBlockRows; b < nb; ++b) s += head[block_off(b) + j];
  }
  c_full[(int64_t)kvh * N + j] = s * ((float)kBlockRows / ((float)G * (float)N));
}

// partial[kvh][slice][c] = sum over the slice's keys, ascending, of C[j] V[j, c]
template <int D>
__global__ void __launch_bounds__(D) exact_semvec_partial_kernel(const float* __restrict__ c_full,
                                                                 const __nv_bfloat16* __restrict__ V, int N, int slices,
                                                                 float* __restrict__ partial) {
  const int kvh = blockIdx.y, sl = blockIdx.x, c = threadIdx.x;
  const int j0 = sl * kSliceKeys, j1 = min(N, j0 + kSliceKeys);
  const float* w = c_full + (int64_t)kvh * N;
  const __nv_bfloat16* v = V + (int64_t)kvh * N * D + c;
  float acc = 0.f;
  for (int j = j0; j < j1; ++j) acc = fmaf(w[j], __bfloat162float(v[(int64_t)j * D]), acc);
  partial[((int64_t)kvh * slices + sl) * D + c] = acc;
}

template <int D>
__global__ void __launch_bounds__(D) exact_semvec_final_kernel(const float* __restrict__ partial, int slices,
                                                               float* __restrict__ sem) {
  const int kvh = blockIdx.x, c = threadIdx.x;
  float acc = 0.f;
  for (int sl = 0; sl < slices; ++sl) acc += partial[((int64_t)kvh * slices + sl) * D + c];
  sem[(int64_t)kvh * D + c] = acc;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

}  // namespace taskkv

using namespace taskkv;

namespace {

struct ExactLayout {
  size_t o_status, o_Cb, o_cfull, o_part, total;
};
// Scratch for batches of hb query heads (a multiple of G).
ExactLayout exact_layout(int64_t hb, int nb, int G, int N, int d, int slices) {
  ExactLayout l;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align256(o + bytes); return at; };
  l.o_status = take(64);
  l.o_Cb = take((size_t)hb * block_off(nb) * 4);
  l.o_cfull = take((size_t)(hb / G) * N * 4);
  l.o_part = take((size_t)(hb / G) * slices * d * 4);
  l.total = o;
  return l;
}

struct ExactShape {
  int N, d, G, nb, slices;
  int64_t q_heads;
  bool ok;
};
ExactShape exact_shape(int32_t n_layers, int32_t n_heads, int32_t n_kv_heads, int32_t head_dim, int32_t seq_len) {
  ExactShape x = {};
  if (n_layers < 1 || n_heads < 1 || n_kv_heads < 1 || n_heads % n_kv_heads != 0) return x;
  if (head_dim != 64 && head_dim != 128) return x;
  if (seq_len < 1 || seq_len > (1 << 20)) return x;
  x.N = seq_len;
  x.d = head_dim;
  x.G = n_heads / n_kv_heads;
  x.nb = (x.N + kBlockRows - 1) / kBlockRows;
  x.slices = (x.N + kSliceKeys - 1) / kSliceKeys;
  x.q_heads = (int64_t)n_layers * n_heads;
  // the longest sequences with many query heads to a KV head are refused: the least a batch can be, one KV group, is then
  // more than 2^28 tiles of 128 rows x 128 keys
  x.ok = (int64_t)x.nb * x.G * ((x.nb + 15) / 16) <= (1 << 24);
  return x;
}
// Most query heads per batch: whole KV groups, as many as a launch takes (grid dimension y of the sums: a KV head each;
// blocks of 128 query rows in one launch of the prefix kernel), scratch within `budget` bytes (0 if not even one group fits).
int64_t exact_heads_per_batch(const ExactShape& x, size_t budget) {
  int64_t hb = x.q_heads;
  hb = std::min<int64_t>(hb, (int64_t)65535 * x.G);
  hb = std::max<int64_t>(x.G, std::min<int64_t>(hb, 0x3fffffff / x.nb / x.G * x.G));
  while (hb > x.G && exact_layout(hb, x.nb, x.G, x.N, x.d, x.slices).total > budget)
    hb = std::max<int64_t>(x.G, hb / 2 / x.G * x.G);
  return exact_layout(hb, x.nb, x.G, x.N, x.d, x.slices).total <= budget ? hb : 0;
}
constexpr size_t kOwnBudget = (size_t)1536 << 20;   // what the library asks the stream's pool for by itself

}  // namespace

extern "C" size_t taskkv_exact_semantic_bytes(int32_t n_layers, int32_t n_heads, int32_t n_kv_heads, int32_t head_dim,
                                              int32_t seq_len) {
  const ExactShape x = exact_shape(n_layers, n_heads, n_kv_heads, head_dim, seq_len);
  if (!x.ok) return 0;
  int64_t hb = exact_heads_per_batch(x, kOwnBudget);
  if (hb == 0) hb = x.G;                              // one KV group is the least a batch can be
  return exact_layout(hb, x.nb, x.G, x.N, x.d, x.slices).total;
}

extern "C" taskkv_status taskkv_exact_semantic(const void* q, const void* k, const void* v, int32_t n_layers,
                                               int32_t n_heads, int32_t n_kv_heads, int32_t head_dim, int32_t seq_len,
                                               float* sem_out, float* c_out, void* workspace_mem,
                                               size_t workspace_bytes, taskkv_stream stream) {
  if (!q || !k || !v || !sem_out) return TASKKV_EINVAL;
  const ExactShape x = exact_shape(n_layers, n_heads, n_kv_heads, head_dim, seq_len);
  if (!x.ok) return TASKKV_EINVAL;
  if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v) & 15) return TASKKV_EINVAL;
  if (workspace_mem && ((uintptr_t)workspace_mem & 255)) return TASKKV_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int N = x.N, d = x.d, G = x.G, nb = x.nb, slices = x.slices;
  const int64_t q_heads = x.q_heads;

  int64_t hb = exact_heads_per_batch(x, workspace_mem ? workspace_bytes : kOwnBudget);
  if (hb == 0 && !workspace_mem) hb = G;
  if (hb == 0) return TASKKV_EALLOC;
  const ExactLayout lay = exact_layout(hb, nb, G, N, d, slices);
  unsigned char* ws = static_cast<unsigned char*>(workspace_mem);
  if (!ws && cudaMallocAsync(reinterpret_cast<void**>(&ws), lay.total, s) != cudaSuccess) {
    cudaGetLastError();
    return TASKKV_EALLOC;
  }

  int32_t* status = reinterpret_cast<int32_t*>(ws + lay.o_status);
  float* Cb = reinterpret_cast<float*>(ws + lay.o_Cb);

  cudaError_t e = cudaMemsetAsync(status, 0, 64, s);
  const size_t es = 2;
  for (int64_t h0 = 0; h0 < q_heads && e == cudaSuccess; h0 += hb) {
    const int64_t hn = std::min<int64_t>(hb, q_heads - h0);          // query heads of this batch (a multiple of G)
    const int64_t kv0 = h0 / G, kvn = hn / G;
    const unsigned char* qb = static_cast<const unsigned char*>(q) + (size_t)h0 * N * d * es;
    const unsigned char* kb = static_cast<const unsigned char*>(k) + (size_t)kv0 * N * d * es;
    const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(v) + (size_t)kv0 * N * d;
    e = launch_prefix_scores(qb, kb, d, (int)hn, G, N, Cb, status, s);
    if (e != cudaSuccess) break;
    float* cf = c_out ? c_out + (size_t)kv0 * N : reinterpret_cast<float*>(ws + lay.o_cfull);
    float* part = reinterpret_cast<float*>(ws + lay.o_part);
    {
      LaunchScope ls(K_EXACT_SUM, s);
      exact_colsum_kernel<<<dim3((unsigned)((N + 255) / 256), (unsigned)kvn), 256, 0, s>>>(Cb, nb, G, N, cf);
    }
    {
      LaunchScope ls(K_EXACT_SUM, s);
      if (d == 64) exact_semvec_partial_kernel<64><<<dim3(slices, (unsigned)kvn), 64, 0, s>>>(cf, vb, N, slices, part);
      else exact_semvec_partial_kernel<128><<<dim3(slices, (unsigned)kvn), 128, 0, s>>>(cf, vb, N, slices, part);
    }
    {
      LaunchScope ls(K_EXACT_SUM, s);
      if (d == 64) exact_semvec_final_kernel<64><<<(unsigned)kvn, 64, 0, s>>>(part, slices, sem_out + (size_t)kv0 * d);
      else exact_semvec_final_kernel<128><<<(unsigned)kvn, 128, 0, s>>>(part, slices, sem_out + (size_t)kv0 * d);
    }
    e = cudaGetLastError();
  }
  int32_t dev_status = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&dev_status, status, 4, cudaMemcpyDeviceToHost, s);
  if (!workspace_mem) cudaFreeAsync(ws, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return TASKKV_ECUDA;
  }
  return dev_status;
}

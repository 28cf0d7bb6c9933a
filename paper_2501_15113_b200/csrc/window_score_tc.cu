// Observation-window scores (Eq. 12, Eq. 13) on the 5th-generation tensor cores, for bf16 inputs and, as sums of products of
// bf16 planes, for fp32 ones.  Kernels for 32, 64 and 128 window rows (G*L); other windows are filled up with zero rows.
//
// The contraction S = Q_win K^T is 2*G*L*d flop per key (32-128 flop per byte of
// K): too much for the CUDA cores next to an HBM-rate K stream, little for
// tcgen05.  Each CTA is a persistent, warp-specialised pipeline:
//   warp 0        TMA producer: K tiles of 128 keys (and the unit's Q rows) into
//                 128-byte-swizzled shared memory, completion on mbarriers
//   warps 1, 6    tcgen05.mma issuers, alternating tiles; accumulators in TMEM (four of
//                 them); tcgen05.commit frees the smem stage and hands the accumulator over
//   warps 2-5, 7-10  two epilogue groups, alternating tiles: tcgen05.ld, softmax arithmetic
//                 in fp32 registers
// (A third epilogue group, with one accumulator per group and a single issuer so that every accumulator
// keeps one issuer and one reader, was measured at the same speed with 128 rows and is not used.)
// Two passes (two launches), as Eq. 13 needs every row's normaliser before rows can be summed:
//   pass 1 (row statistics)  every epilogue warp keeps a running (max, exp-sum) per window row
//     over the keys it sees in a work item and stores it as the warp's own partial; a small
//     kernel folds the partials of a unit.  With up to 64 rows D[key, row] = K Q^T is used (a
//     TMEM lane is a key) and the warp's 32x32 block is transposed through shared memory;
//     with 128 rows the operands are swapped, D[row, key], and a lane owns a row outright.
//   pass 2 (scores)  D[key, row] = K Q^T: a TMEM lane is a key, so
//     C[key] = sum_rows exp2(s - max_row) / Z_row is a sum inside one thread.
// No warp ever waits for another epilogue warp.  Scores are kept in log2 units (scale
// log2(e)/sqrt(d)); exp is one ex2.approx.  Every wait is bounded: on time-out the CTA records
// TASKKV_ETIMEOUT, stops issuing work, releases its TMEM and returns.
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace taskkv {

using namespace tc;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  // (a thread that comes while another is asking waits for the answer)
  static const EncodeTiledFn fn = [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(ptr);
    cudaGetLastError();
    return static_cast<EncodeTiledFn>(nullptr);
  }();
  return fn;
}

// 2-D bf16 tensor [rows_total][d], box of 64 elements x box_rows rows, 128-byte swizzle.
bool make_tensor_map_2d(CUtensorMap* map, const void* base, int d, uint64_t rows_total, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows_total};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tensor_map_units(CUtensorMap* map, const void* base, int d, int rows, uint64_t units, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)units};
  const cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)rows * d * 2};
  const cuuint32_t box[3] = {64u, (cuuint32_t)box_rows, 1u};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

constexpr int kTile = 128;          // keys per tile (UMMA M in pass 2, key sub-tiles in pass 1)
constexpr int kMaxStages = 6;       // K tiles in flight per CTA (the count is fitted to shared memory)
constexpr int kEpiWarps = 8;        // two groups of four epilogue warps, alternating tiles
static_assert(kEpiWarps == kTcParts, "one partial-statistic slot per epilogue warp");
constexpr int kThreads = 352;       // warp 0 producer; 1, 6 MMA issuers; 2-5 and 7-10 epilogue groups
constexpr uint32_t kTmemCols = 512; // four accumulators of up to 128 columns

// fp32 inputs (SPLIT): every element as the sum of three bf16 planes, exactly, whatever the elements beside it are (split8).  A
// score is the sum of six of the nine products of planes; the second plane is at most 2^-8 and the third 2^-17 of the element,
// so the three left out are below 2^-24 of an element's own term, with either sign (2^-27.4 in the mean square).  The leading
// product has an accumulator of its own, since the tensor cores truncate what does not fit an accumulator's 24 bits; the other
// five share one.
// Error of C against 64 bits, six shapes of 40 to 128 rows: 1.0e-7 to 1.4e-7, fp32 on the CUDA cores 1.9e-7 to 2.6e-7; powers of
// two that scale a channel of the keys up and of the queries down (2^-40 to 2^40) change no bit.  (Planes on one grid per row of
// 64 elements, which sum without truncation, are as good for rows whose elements are of one size, but keep the small elements
// beside a large one in fewer bits: 1e-5 for one channel of 2^10, 1e-3 to 1e-2 for one of 2^20.)
// With more than 32 rows (window_score.cu).  Bound by neither pipe nor issue slots, which are 35 % (tensor, 128 rows; 20 % with 64)
// and 38 % busy, but by a stage's way around: the converting warps' loads and arithmetic, the products, the stage given back, with
// room for two stages.  Both passes and their reduction, 32 units of 6001 keys, d = 64: 64 rows 150 us on the CUDA cores, 83 here,
// 128 rows 250 and 93; one layer of 8 x 8000 keys, d = 128: 64 rows 103 and 54, 128 rows 156 and 63.  128 registers a thread (14
// warps are given those of 16), of which a few words spill in the converting warps.  Warps 0 and 11-13 read the fp32 rows and
// write the planes in the producer's place, warp 1 alone issues.
constexpr int kSplitThreads = 448;
constexpr int kCvtWarps = 4;
constexpr int kPlanes = 3;
constexpr int kSmallPairs = 5;      // smallest first
__device__ constexpr int kPairQ[kSmallPairs] = {2, 0, 1, 1, 0};
__device__ constexpr int kPairK[kSmallPairs] = {0, 2, 1, 0, 1};
constexpr float kPlaneMax = 7.2057594e16f;   // 2^56: tiles with a larger element, or an infinite one, are scored in fp32
constexpr int kStageDepth = 8, kStagePitch = kStageDepth + 4;     // floats of a row staged by rescore(): 16-byte writes hit all banks
constexpr int kOddRing = 8;         // tiles whose marks ("not to be had as planes") are kept

// Work items of one launch (one pass over up to kMaxSeq sequences): (sequence, unit, chunk of chunk_keys keys),
// numbered sequence-major, then unit-major: i = item_off[s] + unit * chunks[s] + chunk.  CTA c of a grid of g
// CTAs takes the items c, c + g, c + 2g, ..., fp32 ones c, 2g - 1 - c, 2g + c, ...: a unit's last chunk is short, and with few
// items a CTA some would get nothing but full ones (128 units of 3000 keys, chunks of 2048 and 952: 32 tiles for half of them).
// Short sequences share a launch so that every SM has work.
constexpr int kMaxSeq = 8;
struct TcMaps {
  CUtensorMap k[kMaxSeq];   // [units * N][d] of each sequence
  CUtensorMap q[kMaxSeq];   // [units][window rows][d]
};
struct TcArgs {
  int pass;                 // 1 = row statistics, 2 = scores
  int n_seq;                // sequences in this launch
  int n_local;              // units per sequence (layers * kv heads)
  int chunk_keys;           // keys per work item (multiple of 512)
  int fine;                 // fine parts and items shorter than 2048 keys: pass 1 stores every 512 keys
  int steps;                // items of the busiest CTA
  int u0[kMaxSeq];          // first unit of each sequence
  int N[kMaxSeq];           // sequence length
  int chunks[kMaxSeq];      // work items per unit
  int item_off[kMaxSeq + 1];
};

// Running (max, sum) pairs in log2 units: a <- a + b.
__device__ __forceinline__ void fold_stat(float2& a, const float2 b) {
  if (b.x > -INFINITY) {
    const float M = fmaxf(a.x, b.x);
    a.y = a.y * exp2f(a.x - M) + b.y * exp2f(b.x - M);
    a.x = M;
  }
}

struct Item {
  int seq, lu, ch;
  int N;                    // keys of the unit
  int krow0;                // first row of the unit in the K tensor map
  bool valid;
};
template <bool SPLIT>
__device__ __forceinline__ Item decode_item(const TcArgs& a, int k) {
  Item it;
  const int i = k * (int)gridDim.x + (SPLIT && (k & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
  it.valid = i < a.item_off[a.n_seq];
  it.seq = 0;
#pragma unroll
  for (int s = 1; s < kMaxSeq; ++s)
    if (s < a.n_seq && i >= a.item_off[s]) it.seq = s;
  const int local = it.valid ? i - a.item_off[it.seq] : 0;
  it.lu = local / a.chunks[it.seq];
  it.ch = local % a.chunks[it.seq];
  const int N = a.N[it.seq];
  it.N = N;
  it.krow0 = it.lu * N;
  return it;
}

// Shared-memory plan, made on the host: the Q blocks and the per-warp areas scale with the number of
// window rows; what is left of the 227 KB goes to K stages (an even count, so that each stage is always
// consumed by the same issuer).
struct TcLayout {
  int stages, q_bufs;
  int tile_bytes, q_block_bytes;      // SPLIT: a stage is the planes of 64 elements of a tile's keys
  int off_q, off_stat, off_trans, off_stage, off_bars;
  int total;
};

inline TcLayout make_layout(int D, int rows, bool split) {
  TcLayout l;
  const int KB = D / 64;
  l.tile_bytes = (split ? kPlanes : KB) * kTile * 128;
  l.q_block_bytes = (split ? kPlanes : 1) * KB * rows * 128;
  const int stat = kEpiWarps * rows * (int)sizeof(float2);
  // with 128 rows pass 1 puts the window rows on the TMEM lanes and needs no transposition
  const int trans = rows == 128 ? 0 : kEpiWarps * 32 * 33 * (int)sizeof(float);
  const int stage = split ? kEpiWarps * 32 * kStagePitch * (int)sizeof(float) : 0;
  const int bars = 512;
  const int budget = 232448 - 1024;     // dynamic shared memory of one CTA minus the alignment slack
  auto fit = [&](int q_bufs) { return (budget - q_bufs * l.q_block_bytes - stat - trans - stage - bars) / l.tile_bytes; };
  l.q_bufs = split && fit(2) < 2 ? 1 : 2;
  int stages = fit(l.q_bufs);
  if (stages > kMaxStages) stages = kMaxStages;
  l.stages = split ? stages : stages & ~1;
  l.off_q = l.stages * l.tile_bytes;
  l.off_stat = l.off_q + l.q_bufs * l.q_block_bytes;
  l.off_trans = l.off_stat + stat;
  l.off_stage = l.off_trans + trans;
  l.off_bars = l.off_stage + stage;
  l.total = l.off_bars + bars + 1024;
  return l;
}

// barrier slots
enum : int {
  B_FULL = 0, B_EMPTY = 8, B_QFULL = 16, B_QEMPTY = 18, B_TFULL = 20, B_TEMPTY = 24, B_COUNT = 28
};

// What pass 2 knows of a row: its maximum and the weight 1 / (sum rows), or one offset max + log2(sum) + log2(rows), with which a
// score costs one load and one addition less.  An offset is rounded to 2^-24 of itself: with 64 or 128 rows of bf16 to average
// over that does not show, with up to 32, and beside the error of fp32 scores, it would.
__host__ __device__ constexpr bool stat_pairs(int rows, bool split) { return split || rows == 32; }

// Whether pass 1's items may be shorter than 2048 keys, down to the 512 of one part.  Four times the slots of a row: with 128
// rows a slot is two warps' and there is room; fp32 rows get it (partial_slots), since a tile of theirs takes several times
// as long and a call of few units waits for one CTA's walk over 16 of them (8 units of 2500 keys, 64 rows: 73 us a call
// with 2048, 53 with 512 at d = 64, 98 and 67 at d = 128; on the CUDA cores 56 and 77).
__host__ __device__ constexpr bool fine_parts(int rows, bool split) { return split || rows == 128; }

// `W` (32 or 64) scores of this thread's lane; SPLIT: the sum of the two accumulators.
template <int W, bool SPLIT>
__device__ __forceinline__ void load_scores(uint32_t taddr, uint32_t (&r)[W]) {
  if constexpr (W == 64) tc_ld64(taddr, r);
  else tc_ld32(taddr, r);
  if constexpr (SPLIT) {
    static_assert(W == 32, "the second accumulator's columns take registers, too");
    uint32_t rest[W];
    tc_ld32(taddr + 128u, rest);
    tc_wait_ld();
#pragma unroll
    for (int i = 0; i < W; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(rest[i]));
  } else {
    tc_wait_ld();
  }
}

// Eight elements as three planes of eight bf16: x = b0 + b1 + b2 exactly (for |x| above 2^-100; below, to 2^-126).  Adding x to
// 2^16 x leaves x rounded to a bf16's eight bits behind when 2^16 x is taken away again (Dekker's splitting), the rest of at
// most 16 bits goes the same way, and what is left then has eight.
__device__ __forceinline__ void split8(const float4& lo, const float4& hi, uint4 (&plane)[kPlanes]) {
  float2 v[4] = {make_float2(lo.x, lo.y), make_float2(lo.z, lo.w), make_float2(hi.x, hi.y), make_float2(hi.z, hi.w)};
  const float2 up = make_float2(65536.f, 65536.f), down = make_float2(-65536.f, -65536.f), neg_one = make_float2(-1.f, -1.f);
  uint32_t w[kPlanes][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int pl = 0; pl < kPlanes; ++pl) {
      float2 b = v[i];
      if (pl < kPlanes - 1) {
        b = __ffma2_rn(b, down, __ffma2_rn(b, up, b));
        v[i] = __ffma2_rn(b, neg_one, v[i]);
      }
      w[pl][i] = __byte_perm(__float_as_uint(b.x), __float_as_uint(b.y), 0x7632);
    }
  }
#pragma unroll
  for (int pl = 0; pl < kPlanes; ++pl) plane[pl] = make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
}
// 64 elements of rows of an fp32 matrix (`pitch` floats a row; src: the first of the batch's; rows from `there` on are zeros), by
// the converting warps' threads (thread i), eight elements a thread and row: the c-th four of each half, so that neighbours read
// neighbouring words (which element is where in a row of planes does not matter as long as keys and queries agree).
constexpr int kCvtThreads = kCvtWarps * 32, kBatchRows = kCvtThreads / 8 * 4;
struct Batch { float4 lo[4], hi[4]; };
__device__ __forceinline__ void load_batch(Batch& x, const float* __restrict__ src, int pitch, int there, int i) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int row = (b * kCvtThreads + i) >> 3, c = i & 7;
    x.lo[b] = x.hi[b] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < there) {
      const float4* at = reinterpret_cast<const float4*>(src + (size_t)row * pitch) + c;
      x.lo[b] = at[0];
      x.hi[b] = at[8];
    }
  }
}
// ... as three planes in shared memory, rows of 128 bytes in the 128-byte swizzle, plane_pitch bytes apart (dst: the batch's
// first row, a multiple of eight).  Returns the largest |element| that this thread has (a NaN is not seen; it stays one).
__device__ __forceinline__ float store_batch(const Batch& x, unsigned char* dst, int plane_pitch, int i) {
  float top = 0.f;
#pragma unroll
  for (int b0 = 0; b0 < 4; b0 += 2) {
    uint4 plane[2][kPlanes];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float4 lo = x.lo[b0 + b], hi = x.hi[b0 + b];
      top = fmaxf(top, fmaxf(fmaxf(fmaxf(fabsf(lo.x), fabsf(lo.y)), fmaxf(fabsf(lo.z), fabsf(lo.w))),
                             fmaxf(fmaxf(fabsf(hi.x), fabsf(hi.y)), fmaxf(fabsf(hi.z), fabsf(hi.w)))));
      split8(lo, hi, plane[b]);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int row = ((b0 + b) * kCvtThreads + i) >> 3, c = i & 7;
#pragma unroll
      for (int pl = 0; pl < kPlanes; ++pl)
        *reinterpret_cast<uint4*>(dst + pl * plane_pitch + row * 128 + ((c ^ (row & 7)) << 4)) = plane[b][pl];
    }
  }
  return top;
}
// Asks for `rows` rows (of `bytes` bytes, one after the other) to be brought into L2.
__device__ __forceinline__ void prefetch_rows(const void* src, int rows, int bytes) {
  if (rows > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(rows * bytes) : "memory");
}
// A tile with an element, of its keys or of the queries, that planes do not hold (too large for products and sums to stay finite,
// or infinite itself: products of planes are NaN where the score is infinite): the tile is scored again in fp32, this thread's
// lane against `n` rows of `other`, and put into the accumulators.  A call of its own: a few elements at a time, of the lane's
// row in registers and of 32 other rows in the warp's shared memory (`stage`), from where a load serves all lanes; the next ones
// are on their way meanwhile.  Eight elements, since what the call needs in registers the code around it spills (sixteen: ordinary
// calls 6 to 20 % slower).  32 units of 6001 keys, d = 64, all tiles scored like this, both passes: 64 rows 0.35 ms, 128 rows
// 0.56; on the CUDA cores alone 0.15 and 0.25; with a load of either side from global memory for every product 7.9 and 14.
template <int D>
__device__ __noinline__ void rescore(uint32_t taddr, const float* __restrict__ mine, bool there, const float* __restrict__ other,
                                     int n, int cols, float* stage) {
  constexpr int V = kStageDepth / 4;
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int c0 = 0; c0 < cols && c0 < n; c0 += 32) {
    float sum[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) sum[c] = 0.f;
    const float* theirs = other + (size_t)min(c0 + lane, n - 1) * D;
    float4 m[V], o[V];
#pragma unroll
    for (int i = 0; i < V; ++i) { m[i] = reinterpret_cast<const float4*>(mine)[i]; o[i] = reinterpret_cast<const float4*>(theirs)[i]; }
#pragma unroll 1
    for (int x = 0; x < D; x += kStageDepth) {
      __syncwarp();                                   // the rows staged before have been read
#pragma unroll
      for (int i = 0; i < V; ++i) *reinterpret_cast<float4*>(stage + lane * kStagePitch + 4 * i) = o[i];
      __syncwarp();
      const int next = x + kStageDepth < D ? x + kStageDepth : x;
      float4 m1[V];
#pragma unroll
      for (int i = 0; i < V; ++i) {
        m1[i] = reinterpret_cast<const float4*>(mine + next)[i];
        o[i] = reinterpret_cast<const float4*>(theirs + next)[i];
      }
#pragma unroll
      for (int c = 0; c < 32; ++c) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(stage + c * kStagePitch + 4 * i);
          sum[c] = fmaf(m[i].x, v.x, sum[c]);
          sum[c] = fmaf(m[i].y, v.y, sum[c]);
          sum[c] = fmaf(m[i].z, v.z, sum[c]);
          sum[c] = fmaf(m[i].w, v.w, sum[c]);
        }
      }
#pragma unroll
      for (int i = 0; i < V; ++i) m[i] = m1[i];
    }
    uint32_t r[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) r[c] = there && c0 + c < n ? __float_as_uint(sum[c]) : 0u;
    __syncwarp();
    tc_st32(taddr + (uint32_t)c0, r);
#pragma unroll
    for (int c = 0; c < 32; ++c) r[c] = 0u;
    tc_st32(taddr + 128u + (uint32_t)c0, r);
  }
  tc_wait_st();
}

// ROWS (32, 64 or 128: columns of an accumulator) is a template argument also for the sake of registers: with 128 rows the
// gather of another chunk of layers shares the SMs with this kernel, and how many of its blocks (6144 registers) fit beside
// a CTA is decided here.  One kernel for all row counts took 168 registers a thread, which leaves room for one gather block:
// 7.0 -> 7.5 ms for 32 layers of 131072 keys; this one takes 128, room for three.  FILLED: the window has ROWS rows; the
// masks of the others cost full windows 0.5 us a layer of 8191 keys if they are only known at run time.
template <int D, int ROWS, bool FILLED, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? kSplitThreads : kThreads, 1)
window_tc_kernel(const __grid_constant__ TcMaps maps, DeviceProblem p, const __grid_constant__ TcArgs a,
                 TcLayout lay) {
  constexpr int KB = D / 64;
  constexpr bool PAIR = stat_pairs(ROWS, SPLIT);
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment: the swizzle pattern is a function of the address bits
  // (offset added to the array itself: a round trip through an integer would turn every access below into a
  // generic-address load or store)
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* sK = smem;                                         // [stages][KB][128 keys][128 B]; SPLIT: [stages][planes][128 keys][128 B]
  unsigned char* sQ = smem + lay.off_q;                             // [2][KB][rows][128 B]; SPLIT: [q_bufs][planes][KB][rows][128 B]
  float2* sStat = reinterpret_cast<float2*>(smem + lay.off_stat);   // [8 warps][rows]
  float* sTrans = reinterpret_cast<float*>(smem + lay.off_trans);   // [8 warps][32][33]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + lay.off_bars);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  volatile int* sOdd = s_abort + 1;                                 // [converting warps][kOddRing]  tile not in planes

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int rows = ROWS;                // the window's own rows: p.rows
  const int L = p.L;
  const int S = lay.stages;
  const uint32_t bar0 = smem_u32(bars);
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };

  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(BAR(B_FULL + i), SPLIT ? kCvtWarps : 1); mbar_init(BAR(B_EMPTY + i), 1); }
    for (int i = 0; i < 4; ++i) {
      mbar_init(BAR(B_TFULL + i), 1);
      mbar_init(BAR(B_TEMPTY + i), 4);     // the four warps of the group that reads the accumulator
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(B_QFULL + i), SPLIT ? kCvtWarps : 1);
      mbar_init(BAR(B_QEMPTY + i), SPLIT ? 1 : 2);     // (both) issuers release a Q block
    }
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tc_alloc(smem_u32(s_tmem), kTmemCols);
    tc_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const float scale2 = kLog2e * rsqrtf((float)D);
  grid_dependency_wait();       // the setup above runs under the tail of the kernel before this one

  if (SPLIT && (warp == 0 || warp > 10)) {
    // ------------------------------------------------------------ converting warps.  A stage is two batches of 64 keys; the
    // next batch's loads are on their way while one is converted, and tiles are asked into L2 two ahead.
    const int me = warp == 0 ? 0 : warp - 10, i = me * 32 + lane;
    int stage = 0, qb = 0, n = 0;
    uint32_t phase = 0, qphase[2] = {0, 0};
    bool ok = true;
    auto hand_over = [&](int bar) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(bar));
    };
    for (int k = 0; k < a.steps && ok; ++k) {
      const Item it = decode_item<SPLIT>(a, k);
      if (!it.valid) continue;
      const int u = a.u0[it.seq] + it.lu;
      const int key0 = it.ch * a.chunk_keys, end = min(it.N, key0 + a.chunk_keys);
      const int ntiles = (end - key0 + kTile - 1) / kTile;
      const float* q = static_cast<const float*>(p.q_ptr[u]);
      const float* kp = static_cast<const float*>(p.k_ptr[u]);
      if (i == 0) prefetch_rows(kp + (size_t)key0 * D, min(2 * kTile, end - key0), D * 4);
      constexpr int kQBatches = SPLIT ? ROWS / kBatchRows : 1;
      static_assert(!SPLIT || ROWS % kBatchRows == 0, "the queries' rows are converted in whole batches");
      float q_top = 0.f;
#pragma unroll 1
      for (int x = 0; x < KB * kQBatches; ++x) {
        const int kb = x / kQBatches, r0 = x % kQBatches * kBatchRows;
        Batch qx;
        load_batch(qx, q + (size_t)r0 * D + kb * 64, D, p.rows - r0, i);
        if (x == 0) ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
        if (!ok) break;
        q_top = fmaxf(q_top, store_batch(qx, sQ + (size_t)qb * lay.q_block_bytes + (kb * ROWS + r0) * 128, KB * ROWS * 128, i));
      }
      if (!ok) break;
      hand_over(B_QFULL + qb);
      qphase[qb] ^= 1;
      if (lay.q_bufs == 2) qb ^= 1;
      Batch x0, x1;
      load_batch(x0, kp + (size_t)key0 * D, D, it.N - key0, i);
      float top = q_top;
      for (int c = 0; c < ntiles * KB; ++c) {
        const int t = c / KB, kb = c % KB, at = key0 + t * kTile;
        load_batch(x1, kp + (size_t)(at + kBatchRows) * D + kb * 64, D, it.N - at - kBatchRows, i);
        if (kb == 0 && i == 0) prefetch_rows(kp + (size_t)(at + 2 * kTile) * D, min(kTile, end - at - 2 * kTile), D * 4);
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
        if (!ok) break;
        unsigned char* dst = sK + (size_t)stage * lay.tile_bytes;
        top = fmaxf(top, store_batch(x0, dst, kTile * 128, i));
        const int t1 = (c + 1) / KB, at1 = key0 + t1 * kTile;
        if (c + 1 < ntiles * KB) load_batch(x0, kp + (size_t)at1 * D + (c + 1) % KB * 64, D, it.N - at1, i);
        top = fmaxf(top, store_batch(x1, dst + kBatchRows * 128, kTile * 128, i));
        if (kb == KB - 1) {
          // (the tile whose entry this was is done: its accumulator has been used again since)
          const bool all = __all_sync(0xffffffffu, top < kPlaneMax);
          if (lane == 0) sOdd[me * kOddRing + (n & (kOddRing - 1))] = all ? 0 : 1;
          top = q_top;
          ++n;
        }
        hand_over(B_FULL + stage);
        if (++stage == S) { stage = 0; phase ^= 1; }
      }
    }
    // drain, as below
    for (int j = 0; j < S && ok; ++j) {
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
      if (++stage == S) { stage = 0; phase ^= 1; }
    }
    for (int j = 0; j < lay.q_bufs && ok; ++j, qb = lay.q_bufs == 2 ? qb ^ 1 : qb)
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
  } else if (!SPLIT && warp == 0) {
    // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
    {
      int stage = 0, qb = 0;
      uint32_t phase = 0, qphase[2] = {0, 0};
      bool ok = true;
      for (int k = 0; k < a.steps && ok; ++k) {
        const Item it = decode_item<SPLIT>(a, k);
        if (!it.valid) continue;
        const int N = it.N;
        const int key0 = it.ch * a.chunk_keys;
        const int ntiles = (min(N, key0 + a.chunk_keys) - key0 + kTile - 1) / kTile;
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(BAR(B_QFULL + qb), (uint32_t)lay.q_block_bytes);
          for (int kb = 0; kb < KB; ++kb)
            tma_load_3d(smem_u32(sQ + (size_t)qb * lay.q_block_bytes + (size_t)kb * rows * 128), &maps.q[it.seq],
                        kb * 64, 0, it.lu, BAR(B_QFULL + qb));
        }
        __syncwarp();
        qphase[qb] ^= 1;
        qb ^= 1;
        for (int t = 0; t < ntiles; ++t) {
          ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
          if (!ok) break;
          if (elect_one()) {
            mbar_expect_tx(BAR(B_FULL + stage), (uint32_t)lay.tile_bytes);
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
              tma_load_2d(smem_u32(sK + (size_t)stage * lay.tile_bytes + (size_t)kb * kTile * 128), &maps.k[it.seq],
                          kb * 64, it.krow0 + key0 + t * kTile, BAR(B_FULL + stage));
          }
          __syncwarp();
          if (++stage == S) { stage = 0; phase ^= 1; }
        }
      }
      // Drain: every tcgen05.commit aimed at this CTA's barriers must have arrived before the CTA exits,
      // or it would land on the barriers of the next CTA that is given this shared memory.
      for (int i = 0; i < S && ok; ++i) {
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
        if (++stage == S) { stage = 0; phase ^= 1; }
      }
      for (int i = 0; i < 2 && ok; ++i, qb ^= 1)
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
    }
  } else if (SPLIT && warp == 6) {
  } else if (SPLIT && warp == 1) {
    // ------------------------------------------------------------ MMA issuer for planes: tile n goes to accumulator n & 1,
    // its leading products to columns 256 (n & 1), the others 128 columns on
    int stage = 0, qb = 0, n = 0;
    uint32_t sphase = 0, qphase[2] = {0, 0};
    const uint32_t idesc = instr_desc(128, rows);
    const uint64_t desc_hi = smem_desc(0);
    bool ok = true;
    for (int k = 0; k < a.steps && ok; ++k) {
      const Item it = decode_item<SPLIT>(a, k);
      if (!it.valid) continue;
      const int key0 = it.ch * a.chunk_keys;
      const int ntiles = (min(it.N, key0 + a.chunk_keys) - key0 + kTile - 1) / kTile;
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QFULL + qb), qphase[qb], s_abort));
      if (!ok) break;
      qphase[qb] ^= 1;
      const uint32_t q_lo = smem_u32(sQ + (size_t)qb * lay.q_block_bytes) >> 4;
      const bool swap = a.pass == 1 && rows == 128;   // D[row, key] instead of D[key, row]
      for (int t = 0; t < ntiles && ok; ++t, ++n) {
        const int acc = n & 1;
        const uint32_t d_main = tmem_base + (uint32_t)acc * 256u, d_rest = d_main + 128u;
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_TEMPTY + acc), ((uint32_t)(n >> 1) & 1u) ^ 1u, s_abort));
        for (int kb = 0; kb < KB && ok; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_FULL + stage), sphase, s_abort));
          if (!ok) break;
          tc_fence_after();
          const uint32_t k_lo = smem_u32(sK + (size_t)stage * lay.tile_bytes) >> 4;
          if (elect_one()) {
            auto product = [&](uint32_t d, int pq, int pk, int kk, uint32_t add) {
              const uint64_t kd = desc_hi | (uint64_t)(k_lo + (uint32_t)((pk * kTile * 128 + kk * 32) >> 4));
              const uint64_t qd = desc_hi | (uint64_t)(q_lo + (uint32_t)(((pq * KB + kb) * rows * 128 + kk * 32) >> 4));
              if (swap) tc_mma(d, qd, kd, idesc, add);
              else tc_mma(d, kd, qd, idesc, add);
            };
#pragma unroll
            for (int x = 0; x < kSmallPairs; ++x)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) product(d_rest, kPairQ[x], kPairK[x], kk, (kb | x | kk) ? 1u : 0u);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) product(d_main, 0, 0, kk, (kb | kk) ? 1u : 0u);
            tc_commit(BAR(B_EMPTY + stage));
            if (kb == KB - 1) tc_commit(BAR(B_TFULL + acc));
          }
          __syncwarp();
          if (++stage == S) { stage = 0; sphase ^= 1; }
        }
      }
      if (!ok) break;
      if (elect_one()) tc_commit(BAR(B_QEMPTY + qb));
      __syncwarp();
      if (lay.q_bufs == 2) qb ^= 1;
    }
  } else if (warp == 1 || warp == 6) {
    // ------------------------------------------------------------ MMA issuers: D[key, row] = K Q^T, both passes.
    // Two elected threads: the issue -> commit -> hand-over chain of one tile overlaps with the other's.
    // Tiles are numbered n = 0, 1, ... per CTA across items: issuer n & 1, smem stage n % stages, TMEM
    // accumulator n & 3 (read by epilogue group n & 1).
    // The per-tile bookkeeping is kept to counters that step by two (this issuer's tiles), and the
    // descriptors to one add on a precomputed low word: a lone warp issues an instruction only every few cycles.
    {
      const int me = warp == 1 ? 0 : 1;
      int qb = 0, tiles_before = 0;
      int stage = me, acc = me;                 // S is even: own stages me, me + 2, ...; accumulators me, me + 2
      uint32_t sphase = 0, aphase = 0;
      uint32_t qphase[2] = {0, 0};
      const uint32_t idesc = instr_desc(128, rows);
      const uint64_t desc_hi = smem_desc(0);    // everything but the start address
      bool ok = true;
      for (int k = 0; k < a.steps && ok; ++k) {
        const Item it = decode_item<SPLIT>(a, k);
        if (!it.valid) continue;
        const int N = it.N;
        const int key0 = it.ch * a.chunk_keys;
        const int ntiles = (min(N, key0 + a.chunk_keys) - key0 + kTile - 1) / kTile;
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QFULL + qb), qphase[qb], s_abort));
        if (!ok) break;
        qphase[qb] ^= 1;
        const uint32_t q_lo = smem_u32(sQ + (size_t)qb * lay.q_block_bytes) >> 4;
        const bool swap = a.pass == 1 && rows == 128;   // D[row, key] instead of D[key, row]
        for (int t = (me ^ tiles_before) & 1; t < ntiles; t += 2) {
          ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_FULL + stage), sphase, s_abort) &&
                                           mbar_wait(BAR(B_TEMPTY + acc), aphase ^ 1, s_abort));
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * 128u;
          const uint32_t k_lo = smem_u32(sK + (size_t)stage * lay.tile_bytes) >> 4;
          if (elect_one()) {
#pragma unroll
            for (int kb = 0; kb < KB; ++kb)
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const uint64_t ad = desc_hi | (uint64_t)(k_lo + (uint32_t)((kb * kTile * 128 + k * 32) >> 4));
                const uint64_t bd = desc_hi | (uint64_t)(q_lo + (uint32_t)((kb * rows * 128 + k * 32) >> 4));
                if (swap) tc_mma(d_tmem, bd, ad, idesc, (kb | k) ? 1u : 0u);
                else tc_mma(d_tmem, ad, bd, idesc, (kb | k) ? 1u : 0u);
              }
            tc_commit(BAR(B_EMPTY + stage));   // smem stage free once these MMAs have read it
            tc_commit(BAR(B_TFULL + acc));     // accumulator ready for the epilogue
          }
          __syncwarp();
          stage += 2;
          if (stage >= S) { stage -= S; sphase ^= 1; }
          acc ^= 2;
          if (acc == me) aphase ^= 1;
        }
        if (!ok) break;
        tiles_before += ntiles;
        if (elect_one()) tc_commit(BAR(B_QEMPTY + qb));   // this issuer is done with the Q block
        __syncwarp();
        qb ^= 1;
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue: two groups of 4 warps (2-5 take
    // even tiles, 7-10 odd tiles); a TMEM lane is a key
    const int ew = warp < 6 ? warp - 2 : warp - 3;  // 0..7
    const int grp = ew >> 2;
    const int quad = warp & 3;                      // TMEM lane quadrant this warp may read
    float* myStat = reinterpret_cast<float*>(sStat) + ew * 2 * rows;
    float* myT = sTrans + ew * (32 * 33);
    constexpr int kWide = SPLIT ? 32 : 64;          // columns per tensor-memory load where many are to be had
    int n = 0;
    bool ok = true;
    // pass 2: the rows' pairs or offsets (which turn a raw score into its share of C) of a unit, lane i holding rows i, i + 32,
    // ...; loaded one item ahead
    const float* stat_g = p.stat;
    float pre[4], pre_w[PAIR ? 4 : 1];
    auto fetch_stats = [&](int k) {
      const Item nx = decode_item<SPLIT>(a, k);
      const float* st = stat_g + (size_t)(a.u0[nx.seq] + nx.lu) * (2 * p.rows_pad);
#pragma unroll
      for (int q = 0; q < 4; ++q) {               // a row that is not there weighs nothing
        if (q * 32 >= rows) break;
        const bool there = nx.valid && q * 32 + lane < p.rows;
        pre[q] = there ? st[q * 32 + lane] : PAIR ? 0.f : INFINITY;
        if (PAIR) pre_w[PAIR ? q : 0] = there ? st[p.rows_pad + q * 32 + lane] : 0.f;
      }
    };
    if (a.pass == 2) fetch_stats(0);
    for (int k = 0; k < a.steps && ok; ++k) {
      const Item it = decode_item<SPLIT>(a, k);
      if (!it.valid) continue;
      const int u = a.u0[it.seq] + it.lu;
      const int N = it.N;
      const int key0 = it.ch * a.chunk_keys;
      const int ntiles = (min(N, key0 + a.chunk_keys) - key0 + kTile - 1) / kTile;
      // pass 1 state: after the transposition lane = window row (rg * 32 + lane); raw (unscaled) maxima
      float m_run[4], z_run[4];
#pragma unroll
      for (int rg = 0; rg < 4; ++rg) { m_run[rg] = -INFINITY; z_run[rg] = 0.f; }
      if (a.pass == 2) {
        __syncwarp();                       // the previous item's readers of myStat are done
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q * 32 < rows) {
            myStat[q * 32 + lane] = pre[q];
            if (PAIR) myStat[rows + q * 32 + lane] = pre_w[PAIR ? q : 0];
          }
        __syncwarp();
        fetch_stats(k + 1);                 // in flight while this item's tiles are worked on
      }
      // Which of the item's tiles this group takes depends on how many tiles the CTA has seen before (n): with n even
      // at the item's start it is the even ones.  The partial statistics below are filed under that parity, not under
      // the group, so that a slot always holds the same tiles (and keys) whatever else the CTA worked on before:
      // results do not depend on how a problem is cut into launches -- nor on the length of the items: what is stored
      // covers 16 tiles of the unit, and with fine parts those are folded from four parts of 4 tiles each, here (long
      // items) or, where items are shorter than 16 tiles (a.fine), from the stored parts by the reduction.
      const int par = grp ^ (n & 1);                 // parity, within the item, of the tiles this warp takes
      constexpr int sub_shift = fine_parts(ROWS, SPLIT) ? 2 : 4;     // log2 of the tiles per part
      int sub = 0;                                   // the part this warp is working on, counted from the item's first
      constexpr int kGroupRows = ROWS == 128 ? 1 : ROWS / 32;        // rows of this lane
      float2 group[kGroupRows];
#pragma unroll
      for (int rg = 0; rg < kGroupRows; ++rg) group[rg] = make_float2(-INFINITY, 0.f);
      auto end_part = [&]() {
        // slot (part of the unit, part of the warps): (tile parity, lane quadrant); with 128 rows a quadrant is a set of
        // rows, so there it is the tile parity alone
        float2* base = reinterpret_cast<float2*>(p.stat_part) + (size_t)u * p.chunks_max * p.rows_pad;
        const int tile0 = key0 / kTile;
        const bool last = (sub & 3) == 3 || sub == ((ntiles + 3) >> 2) - 1;
#pragma unroll
        for (int rg = 0; rg < kGroupRows; ++rg) {
          const int row = (rows == 128 ? quad : rg) * 32 + lane;
          const int slots = rows == 128 ? 2 : kTcParts, slot = rows == 128 ? par : par * 4 + quad;
          float2 mine = make_float2(m_run[rg] * scale2, z_run[rg]);
          int part = (tile0 >> sub_shift) + sub;
          if (fine_parts(ROWS, SPLIT) && !a.fine) {
            fold_stat(group[rg], mine);
            if (!last) continue;
            mine = group[rg];
            group[rg] = make_float2(-INFINITY, 0.f);
            part = (tile0 >> 4) + (sub >> 2);
          }
          if (row < p.rows) base[(size_t)(part * slots + slot) * p.rows_pad + row] = mine;
        }
#pragma unroll
        for (int rg = 0; rg < 4; ++rg) { m_run[rg] = -INFINITY; z_run[rg] = 0.f; }
        ++sub;
      };
      for (int t = 0; t < ntiles; ++t, ++n) {
        if ((n & 1) != grp) continue;
        if (a.pass == 1 && (t >> sub_shift) != sub) end_part();
        const int acc = SPLIT ? n & 1 : n & 3;
        const uint32_t accphase = (uint32_t)((SPLIT ? n >> 1 : n >> 2) & 1);
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_TFULL + acc), accphase, s_abort));
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * (SPLIT ? 256u : 128u);
        const int tbase = key0 + t * kTile;
        if constexpr (SPLIT) {
          int odd = 0;
#pragma unroll
          for (int w = 0; w < kCvtWarps; ++w) odd |= sOdd[w * kOddRing + (n & (kOddRing - 1))];
          if (odd) {
            // lane and column: row and key in pass 1 of 128 rows, key and row otherwise
            const float* q = static_cast<const float*>(p.q_ptr[u]);
            const float* kp = static_cast<const float*>(p.k_ptr[u]);
            const int l = quad * 32 + lane;
            const bool swap = a.pass == 1 && rows == 128;
            const bool there = swap ? l < p.rows : tbase + l < N;
            const float* mine = swap ? q + (size_t)(there ? l : 0) * D : kp + (size_t)(there ? tbase + l : 0) * D;
            rescore<D>(taddr, mine, there, swap ? kp + (size_t)tbase * D : q, swap ? min(kTile, N - tbase) : p.rows, swap ? kTile : rows,
                       reinterpret_cast<float*>(smem + lay.off_stage) + ew * (32 * kStagePitch));
          }
        }
        const bool tail = (tbase + kTile - 1 > N - L);   // some key of the tile is masked for some row
        if (a.pass == 1 && rows == 128) {
          // a TMEM lane is a window row (quad * 32 + lane), the 128 columns are the keys of the tile
          const int pos = N - L + ((quad * 32 + lane) % L);   // last key this window row may see
#pragma unroll
          for (int cg = 0; cg < kTile / kWide; ++cg) {   // kWide keys per TMEM load
            uint32_t r[kWide];
            load_scores<kWide, SPLIT>(taddr + (uint32_t)(cg * kWide), r);
            float x[kWide];
            if (!tail) {
#pragma unroll
              for (int k = 0; k < kWide; ++k) x[k] = __uint_as_float(r[k]);
            } else {
#pragma unroll
              for (int k = 0; k < kWide; ++k) {
                const int j = tbase + cg * kWide + k;
                x[k] = (j <= pos && j < N) ? __uint_as_float(r[k]) : -INFINITY;
              }
            }
            float cm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int k = 0; k < kWide; ++k) cm4[k & 3] = fmaxf(cm4[k & 3], x[k]);
            const float cm = fmaxf(fmaxf(cm4[0], cm4[1]), fmaxf(cm4[2], cm4[3]));
            if (cm > m_run[0]) {
              z_run[0] *= ex2((m_run[0] - cm) * scale2);
              m_run[0] = cm;
            }
            if (m_run[0] > -INFINITY) {
              const float ms = -m_run[0] * scale2;
              float zs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
              for (int k = 0; k < kWide; ++k) zs[k & 3] += ex2(fmaf(x[k], scale2, ms));
              z_run[0] += (zs[0] + zs[1]) + (zs[2] + zs[3]);
            }
          }
        } else if (a.pass == 1) {
          const int jw = tbase + quad * 32;              // first key of this warp's 32 lanes
#pragma unroll
          for (int rg = 0; rg < 4; ++rg) {
            if (rg * 32 < rows) {
              uint32_t r[32];
              load_scores<32, SPLIT>(taddr + (uint32_t)(rg * 32), r);
              // transpose the warp's [32 keys][32 rows] block through shared memory
#pragma unroll
              for (int c = 0; c < 32; ++c) myT[lane * 33 + c] = __uint_as_float(r[c]);
              __syncwarp();
              float x[32];
              if (!tail) {
#pragma unroll
                for (int k = 0; k < 32; ++k) x[k] = myT[k * 33 + lane];
              } else {
                const int pos = N - L + ((rg * 32 + lane) % L);   // last key this window row may see
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                  const int j = jw + k;
                  x[k] = (j <= pos && j < N) ? myT[k * 33 + lane] : -INFINITY;
                }
              }
              __syncwarp();
              // four interleaved chains: a single running max / sum would serialise on the ALU latency
              float cm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
              for (int k = 0; k < 32; ++k) cm4[k & 3] = fmaxf(cm4[k & 3], x[k]);
              const float cm = fmaxf(fmaxf(cm4[0], cm4[1]), fmaxf(cm4[2], cm4[3]));
              if (cm > m_run[rg]) {
                z_run[rg] *= ex2((m_run[rg] - cm) * scale2);
                m_run[rg] = cm;
              }
              if (m_run[rg] > -INFINITY) {
                const float ms = -m_run[rg] * scale2;
                float zs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < 32; ++k) zs[k & 3] += ex2(fmaf(x[k], scale2, ms));
                z_run[rg] += (zs[0] + zs[1]) + (zs[2] + zs[3]);
              }
            }
          }
        } else {
          const int j = tbase + quad * 32 + lane;   // this thread's key
          float cs[4] = {0.f, 0.f, 0.f, 0.f};   // four interleaved chains (FMA latency)
          // A row that the window does not have is a zero query, and its score at a key with an infinite element is NaN:
          // such rows are left out, not given a weight of zero.
          if (rows >= 64 && !tail && FILLED) {
            // 64 columns per TMEM load: half the load / wait round trips of the 32-column walk below
            for (int c0 = 0; c0 < rows; c0 += kWide) {
              uint32_t r[kWide];
              load_scores<kWide, SPLIT>(taddr + (uint32_t)c0, r);
              const float4* st4 = reinterpret_cast<const float4*>(myStat + c0);   // four rows per 16-byte load
              const float4* wt4 = reinterpret_cast<const float4*>(myStat + rows + c0);
#pragma unroll
              for (int c = 0; c < kWide; c += 4) {
                const float4 off = st4[c >> 2];
                const float e0 = ex2(fmaf(__uint_as_float(r[c]), scale2, -off.x));
                const float e1 = ex2(fmaf(__uint_as_float(r[c + 1]), scale2, -off.y));
                const float e2 = ex2(fmaf(__uint_as_float(r[c + 2]), scale2, -off.z));
                const float e3 = ex2(fmaf(__uint_as_float(r[c + 3]), scale2, -off.w));
                if constexpr (PAIR) {
                  const float4 w = wt4[c >> 2];
                  cs[0] = fmaf(e0, w.x, cs[0]);
                  cs[1] = fmaf(e1, w.y, cs[1]);
                  cs[2] = fmaf(e2, w.z, cs[2]);
                  cs[3] = fmaf(e3, w.w, cs[3]);
                } else {
                  cs[0] += e0;
                  cs[1] += e1;
                  cs[2] += e2;
                  cs[3] += e3;
                }
              }
            }
          } else if (rows == 32) {
            uint32_t r[32];
            load_scores<32, SPLIT>(taddr, r);
            const float4* mx4 = reinterpret_cast<const float4*>(myStat);
            const float4* wt4 = reinterpret_cast<const float4*>(myStat + rows);
            uint32_t vm = FILLED ? 0xffffffffu : (1u << p.rows) - 1u;   // bit c: window row c sees this thread's key
            if (tail) {
              const int need = j < N ? j - (N - L) : L;        // the residue c % L the row must reach (L: none does)
              int res = 0;
              uint32_t seen = 0;
#pragma unroll
              for (int c = 0; c < 32; ++c) {
                seen |= (uint32_t)(need <= res) << c;
                res = (res + 1 == L) ? 0 : res + 1;
              }
              vm &= seen;
            }
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
              const float4 mx = mx4[c >> 2], w = wt4[c >> 2];
              const float m4[4] = {mx.x, mx.y, mx.z, mx.w}, w4[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float e = ex2(fmaf(__uint_as_float(r[c + i]), scale2, -m4[i]));
                cs[i] = fmaf((vm >> (c + i)) & 1u ? e : 0.f, w4[i], cs[i]);
              }
            }
          } else
          for (int c0 = 0; c0 < (FILLED ? rows : p.rows); c0 += 32) {
            uint32_t r[32];
            load_scores<32, SPLIT>(taddr + (uint32_t)c0, r);
            if (!tail) {
              const float4* st4 = reinterpret_cast<const float4*>(myStat + c0);   // four rows per 16-byte load
              const float4* wt4 = reinterpret_cast<const float4*>(myStat + rows + c0);
#pragma unroll
              for (int c = 0; c < 32; c += 4) {
                const float4 off = st4[c >> 2], w = PAIR ? wt4[c >> 2] : make_float4(1.f, 1.f, 1.f, 1.f);
                const float o4[4] = {off.x, off.y, off.z, off.w}, w4[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  if (FILLED || c0 + c + i < p.rows) {
                    const float e = ex2(fmaf(__uint_as_float(r[c + i]), scale2, -o4[i]));
                    cs[i] = PAIR ? fmaf(e, w4[i], cs[i]) : cs[i] + e;
                  }
              }
            } else {
              // window row c0 + c sees keys up to N - L + (c0 + c) % L.  The residue is counted along (one
              // division per 32 rows): a division per element made this tile cost fourteen ordinary ones
              int res = c0 % L;
              const int need = j - (N - L);         // the row's residue must reach this for key j to be visible
#pragma unroll
              for (int c = 0; c < 32; ++c) {
                const float off = myStat[c0 + c];
                const bool vis = (j < N) && (need <= res) && (FILLED || c0 + c < p.rows);
                if (vis) {
                  const float e = ex2(fmaf(__uint_as_float(r[c]), scale2, -off));
                  cs[c & 3] = PAIR ? fmaf(e, myStat[rows + c0 + c], cs[c & 3]) : cs[c & 3] + e;
                }
                res = (res + 1 == L) ? 0 : res + 1;
              }
            }
          }
          const float csum = (cs[0] + cs[1]) + (cs[2] + cs[3]);
          if (j < N) p.C[p.c_off[u] + j] = csum;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_TEMPTY + acc));
      }
      if (!ok) break;
      if (a.pass == 1) {
        // the last part, and an empty one should it hold no tile of this group
        const int subs = (ntiles + (1 << sub_shift) - 1) >> sub_shift;
        while (sub < subs) end_part();
      }
    }
  }

  // ---------------------------------------------------------------- teardown
  // after a time-out give copies and MMAs still in flight a bounded time to land before the memory is released
  if (*s_abort)
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tc_dealloc(tmem_base, kTmemCols);
  }
  if (tid == 0 && *s_abort) set_status(p.status, TASKKV_ETIMEOUT);
}

// Folds the partial statistics of one unit -> a pair or an offset per row.  One block per unit; 8 to 32 threads share a row, each
// taking every 8th to 32nd slot in order with four loads ahead of the dependent updates, and their results are
// joined in order: the outcome depends on the unit's own length alone.
__global__ void __launch_bounds__(1024) window_tc_reduce_kernel(DeviceProblem p, UnitRange ur, int fine, int pairs) {
  __shared__ float2 tmp[1024];
  const int u = ur.unit(blockIdx.x);
  const int N = p.unit_N[u];
  const int rows = tc_rows(p.rows), P = 1024 / rows;
  const int per = rows == 128 ? 2 : kTcParts;          // warps (or pairs of them) that a part has a slot for
  const int slots = (N + 16 * kTile - 1) / (16 * kTile) * per;
  const int row = threadIdx.x % rows, part = threadIdx.x / rows;
  const float2* src = reinterpret_cast<const float2*>(p.stat_part) + (size_t)u * p.chunks_max * p.rows_pad + row;
  float2 acc = make_float2(-INFINITY, 0.f);
  const bool there = row < p.rows;
  grid_dependency_wait();
  if (!there) {
  } else if (fine) {
    // slot (group, warps) is folded from up to four stored parts
    const int parts = (N + 4 * kTile - 1) / (4 * kTile);
    for (int c = part; c < slots; c += P) {
      float2 o[4], g = make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int q = c / per * 4 + i;
        o[i] = q < parts ? src[(size_t)(q * per + c % per) * p.rows_pad] : make_float2(-INFINITY, 0.f);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) fold_stat(g, o[i]);
      fold_stat(acc, g);
    }
  } else {
    for (int c = part; c < slots; c += 4 * P) {
      float2 o[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        o[i] = c + i * P < slots ? src[(size_t)(c + i * P) * p.rows_pad] : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int i = 0; i < 4; ++i) fold_stat(acc, o[i]);
    }
  }
  tmp[threadIdx.x] = acc;
  __syncthreads();
  if (part == 0 && there) {
    for (int q = 1; q < P; ++q) fold_stat(acc, tmp[q * rows + row]);
    float* st = p.stat + (size_t)u * (2 * p.rows_pad);
    if (pairs) {
      st[row] = acc.y > 0.f ? acc.x : 0.f;
      st[p.rows_pad + row] = acc.y > 0.f ? 1.0f / (acc.y * (float)p.rows) : 0.f;
    } else {
      st[row] = acc.y > 0.f ? acc.x + log2f(acc.y) + log2f((float)p.rows) : INFINITY;
    }
  }
}

// Keys per work item.  Every item costs a Q load and, in pass 2, a statistics load, so long items are better as long as
// the CTAs still get a dozen items each; a launch with fewer takes shorter ones, down to the 512 keys of one partial
// (2048 in pass 1 without fine parts), so that a single layer of a short prompt still reaches every SM: 8 units of
// 8191 keys, 128 rows, took 23.2 us a pass on 32 CTAs of 16 tiles, 15.3 on 128 of 4.
inline int pick_chunk(int64_t units_times_keys, int n_sm, int least) {
  if (units_times_keys / 4096 >= (int64_t)12 * n_sm) return 4096;
  int chunk = 2048;
  while (chunk > least && units_times_keys / chunk < (int64_t)3 * n_sm) chunk /= 2;
  return chunk;
}

template <int D, int ROWS, bool FILLED, bool SPLIT>
cudaError_t launch_tc_d(const DeviceProblem& p, const WindowHostInfo& h, cudaStream_t s, int layer0, int n_layers) {
  const int n_sm = sm_count();
  constexpr int rows = ROWS;
  const TcLayout lay = make_layout(D, rows, SPLIT);
  if (lay.stages < 2) return cudaErrorInvalidValue;
  const int smem = lay.total;
  cudaError_t e = cudaFuncSetAttribute(window_tc_kernel<D, ROWS, FILLED, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int per_seq_all = p.R * p.n_kv;
  const int first = layer0 * p.n_kv;               // the launch covers units [first, first + per_seq) of every sequence
  const int per_seq = n_layers * p.n_kv;
  const int skip = (layer0 - h.base_layer) * p.n_kv;   // units between what h.q / h.k point at and the first one
  if (per_seq <= 0) return cudaSuccess;
  // up to kMaxSeq sequences per pair of launches
  for (int b0 = 0; b0 < h.batch; b0 += kMaxSeq) {
    const int nb = h.batch - b0 < kMaxSeq ? h.batch - b0 : kMaxSeq;
    TcMaps maps;
    if (SPLIT) maps = TcMaps{};                              // fp32 rows are read through the units' pointers
    TcArgs a;
    int64_t keys = 0;
    for (int i = 0; i < nb; ++i) keys += (int64_t)per_seq * h.seq_lens[b0 + i];
    a.n_seq = nb;
    a.n_local = per_seq;
    for (int i = 0; i < kMaxSeq; ++i) {
      const int b = b0 + (i < nb ? i : 0);                  // unused slots repeat the first sequence
      const int N = h.seq_lens[b];
      if (SPLIT) {
      } else if (i >= nb) {
        maps.k[i] = maps.k[0];
        maps.q[i] = maps.q[0];
      } else {
        const char* kb = static_cast<const char*>(h.k[b]) + (size_t)skip * (size_t)N * D * sizeof(__nv_bfloat16);
        const char* qb = static_cast<const char*>(h.q[b]) + (size_t)skip * p.rows * D * sizeof(__nv_bfloat16);
        if (!make_tensor_map_2d(&maps.k[i], kb, D, (uint64_t)per_seq * (uint64_t)N, kTile)) return cudaErrorUnknown;
        if (!make_tensor_map_units(&maps.q[i], qb, D, p.rows, (uint64_t)per_seq, rows)) return cudaErrorUnknown;
      }
      a.u0[i] = b * per_seq_all + first;
      a.N[i] = N;
    }
    auto launch_pass = [&](int pass, int least) -> cudaError_t {
      a.pass = pass;
      a.chunk_keys = pick_chunk(keys, n_sm, least);
      a.fine = pass == 1 && fine_parts(ROWS, SPLIT) && a.chunk_keys < 16 * kTile ? 1 : 0;
      a.item_off[0] = 0;
      for (int i = 0; i < kMaxSeq; ++i) {
        a.chunks[i] = (a.N[i] + a.chunk_keys - 1) / a.chunk_keys;
        a.item_off[i + 1] = a.item_off[i] + (i < nb ? per_seq * a.chunks[i] : 0);
      }
      const int items = a.item_off[nb], grid = items < n_sm ? items : n_sm;
      a.steps = (items + grid - 1) / grid;
      LaunchScope ls(K_WINDOW_TC, s);
      return launch_dependent_smem(window_tc_kernel<D, ROWS, FILLED, SPLIT>, (unsigned)grid, SPLIT ? kSplitThreads : kThreads, (size_t)smem, s,
                                  maps, p, a, lay);
    };
    if (h.lse) {
      // the caller already has the rows' normalisers: no pass 1
      const size_t lse_skip = (size_t)(layer0 - h.base_layer) * p.n_heads * p.L;
      for (int i = 0; i < nb; ++i) {
        e = launch_lse_to_stat(p, (b0 + i) * per_seq_all + first, per_seq,
                               static_cast<const float*>(h.lse[b0 + i]) + lse_skip, stat_pairs(ROWS, SPLIT) ? LSE_PAIR : LSE_OFFSET, s);
        if (e != cudaSuccess) return e;
      }
    } else {
      e = launch_pass(1, fine_parts(ROWS, SPLIT) ? 4 * kTile : kTcChunk);
      if (e != cudaSuccess) return e;
      LaunchScope ls(K_WINDOW_REDUCE, s);
      const UnitRange ur{b0 * per_seq_all + first, per_seq, per_seq_all, nb * per_seq};
      e = launch_dependent(window_tc_reduce_kernel, (unsigned)(nb * per_seq), 1024, s, p, ur, a.fine, stat_pairs(ROWS, SPLIT) ? 1 : 0);
      if (e != cudaSuccess) return e;
    }
    e = launch_pass(2, 4 * kTile);
    if (e != cudaSuccess) return e;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int ROWS, bool SPLIT>
cudaError_t launch_tc_rows(const DeviceProblem& p, const WindowHostInfo& h, cudaStream_t s, int layer0, int n_layers) {
  if (p.rows == ROWS)
    return p.d == 64 ? launch_tc_d<64, ROWS, true, SPLIT>(p, h, s, layer0, n_layers)
                     : launch_tc_d<128, ROWS, true, SPLIT>(p, h, s, layer0, n_layers);
  return p.d == 64 ? launch_tc_d<64, ROWS, false, SPLIT>(p, h, s, layer0, n_layers)
                   : launch_tc_d<128, ROWS, false, SPLIT>(p, h, s, layer0, n_layers);
}
}  // namespace

bool window_tc_supported(const DeviceProblem& p, int dtype) {
  return dtype == TASKKV_BF16 && p.rows <= 128 && encode_fn() != nullptr;
}

cudaError_t launch_window_scores_tc(const DeviceProblem& p, int dtype, const WindowHostInfo& h, cudaStream_t s, int layer0,
                                    int n_layers) {
  if (n_layers < 0) { layer0 = 0; n_layers = p.R; }
  if (dtype == TASKKV_F32)
    return p.rows <= 64 ? launch_tc_rows<64, true>(p, h, s, layer0, n_layers) : launch_tc_rows<128, true>(p, h, s, layer0, n_layers);
  // 32 window rows and sequences short enough for a unit's scores to stay in tensor memory: K is read once
  if (window_res_supported(p, h)) return launch_window_scores_res(p, h, s, layer0, n_layers);
  switch (tc_rows(p.rows)) {
    case 32: return launch_tc_rows<32, false>(p, h, s, layer0, n_layers);
    case 64: return launch_tc_rows<64, false>(p, h, s, layer0, n_layers);
    default: return launch_tc_rows<128, false>(p, h, s, layer0, n_layers);
  }
}

}  // namespace taskkv

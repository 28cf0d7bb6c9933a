// Column sums of the full causal attention matrix in 128-row blocks (Eq. 1-2), for the exact semantic vector: block b
// of a query head is its 128 query rows [128 b, 128 b + 128), which see the first 128 (b + 1) keys of the KV head, and
//   C_b[j] = (1/128) sum_{i in block b} softmax_i[j].
// A CTA owns a block: it walks the block's key tiles twice, first for the rows' normalisers, then, with them, for the
// column sums, so that nothing is exchanged between CTAs and the second walk finds its keys in L2.
//   warp 0          TMA producer: K tiles of 128 keys (four stages), the block's Q rows (two buffers, one block ahead)
//   warps 1, 6      tcgen05.mma issuers, alternate tiles; four accumulators of 128 columns in TMEM
//   warps 2-5, 7-18 four epilogue groups, every fourth tile each
// First walk: D[row, key] = Q K^T, a TMEM lane is a query row and keeps its own running (max, sum); the four groups'
// pairs meet in shared memory.  Second walk: D[key, row] = K Q^T, a lane is a key and sums its column.
// Two exponentials per score at 16 a cycle and SM are 2048 cycles per tile and block on the special-function unit, so a quarter of
// them is computed on the FMA pipe.  That unit is then 67 % busy and the tensor pipe 43 %; what the warps wait for most is their
// tensor-memory loads, one 32-column step after the other, and each other.
// Blocks are dealt out longest first, in both directions alternately, so that every CTA gets the same number of tiles;
// the heads go in groups whose keys fit well into L2.  32 heads x 16384 rows, d = 128, both walks: as two launches of
// the window kernel over (block, 2048 keys) items 4.19 ms (a CTA met the same two of a block's eight key ranges again
// and again, a third more tiles for some than on average), like this with two epilogue groups 2.98 ms, with four 2.76 ms:
// with two warps to a scheduler the special-function unit idles while they hand over.  With the exponentials shared 2.82 -> 2.62 ms
// for a call by itself, 2.91 -> 2.84 in a row of calls, which the power limit slows down (weight2).
#include <cuda.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace taskkv {

using namespace tc;

namespace {

constexpr int kTile = 128;          // keys per tile, query rows per block
constexpr int kStages = 4;          // K tiles in flight (even: a stage always has the same issuer)
constexpr int kGroups = 4;          // epilogue groups of four warps, one per accumulator
constexpr int kEpiWarps = 4 * kGroups;
constexpr int kThreads = (3 + kEpiWarps) * 32;
constexpr int kCols = 32;           // accumulator columns per tensor-memory load
constexpr uint32_t kTmemCols = 512;

struct PrefixMaps {
  CUtensorMap k;                    // [heads / group * N][d]
  CUtensorMap q;                    // [heads * N][d]
};
struct PrefixArgs {
  int N, nb;                        // sequence length, blocks per head
  int heads, group;                 // query heads, query heads per KV head
  int team;                         // query heads that go together (whole KV groups)
  int items, steps;                 // blocks in all, blocks of the busiest CTA
  float* scores;                    // [heads][64 nb (nb + 1)]: block b of a head starts at 64 b (b + 1)
  int32_t* status;
};

struct Block { int head, b; bool valid; };
__device__ __forceinline__ Block block_of(const PrefixArgs& a, int k) {
  const int g = (int)gridDim.x, c = (int)blockIdx.x;
  const int i = k * g + ((k & 1) ? g - 1 - c : c);
  Block x;
  x.valid = i < a.items;
  const int j = x.valid ? i : 0;
  const int per_team = a.team * a.nb;
  const int t = j / per_team, r = j - t * per_team;
  const int members = min(a.team, a.heads - t * a.team);
  const int lvl = r / members;
  x.head = t * a.team + (r - lvl * members);
  x.b = a.nb - 1 - lvl;
  return x;
}

struct PrefixLayout {
  int tile_bytes, off_q, off_stat, off_off, off_bars, total;
};
inline PrefixLayout make_prefix_layout(int D) {
  PrefixLayout l;
  l.tile_bytes = D / 64 * kTile * 128;
  l.off_q = kStages * l.tile_bytes;
  l.off_stat = l.off_q + 2 * l.tile_bytes;
  l.off_off = l.off_stat + 2 * kGroups * kTile * (int)sizeof(float2);
  l.off_bars = l.off_off + kEpiWarps * kTile * (int)sizeof(float);
  l.total = l.off_bars + 512 + 1024;
  return l;
}

__device__ __forceinline__ float2 pair_of(const uint32_t* r, int i) {
  return make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1]));
}
// Weights of columns i, i + 1 of a tile.  Every fourth pair goes through the FMA pipe: the special-function unit alone is
// busy for 1024 of a tile's cycles.  32 heads x 16384 rows, none / 2 / 4 / 5 / 6 / 8 of 16 pairs: 2.82 / 2.64 / 2.62 / 2.68 /
// 2.71 / 2.92 ms for a call by itself (2.89 with the pairs' products and sums unpacked), and 2.91 / 2.84 / 2.84 / 2.89 / - /
// 3.16 (2.98) in a row of calls, which the power limit slows down; the error against 64 bits stays where it was.
constexpr int kFmaEvery = 4;
__device__ __forceinline__ float2 weight2(int i, float2 x) {
  if ((i >> 1) % kFmaEvery == 0) return ex2_fma(x);
  return make_float2(ex2(x.x), ex2(x.y));
}

enum : int {
  B_FULL = 0, B_EMPTY = 4, B_QFULL = 8, B_QEMPTY = 10, B_TFULL = 12, B_TEMPTY = 16, B_STAT = 20, B_COUNT = 22
};

// RAGGED: the last block of a head has fewer than 128 rows.  (A template argument, since the code for such blocks costs the whole
// ones 0.5 to 1 % in the same kernel.)
template <int D, bool RAGGED>
__global__ void __launch_bounds__(kThreads, 1)
prefix_score_kernel(const __grid_constant__ PrefixMaps maps, const __grid_constant__ PrefixArgs a, PrefixLayout lay) {
  constexpr int KB = D / 64;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* sK = smem;                                         // [stages][KB][128 keys][128 B]
  unsigned char* sQ = smem + lay.off_q;                             // [2][KB][128 rows][128 B]
  float2* sStat = reinterpret_cast<float2*>(smem + lay.off_stat);   // [2 blocks][groups][128 rows]
  float* sOff = reinterpret_cast<float*>(smem + lay.off_off);       // [epilogue warps][128 rows]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + lay.off_bars);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + B_COUNT);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar0 = smem_u32(bars);
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(BAR(B_FULL + i), 1); mbar_init(BAR(B_EMPTY + i), 1); }
    for (int i = 0; i < 4; ++i) { mbar_init(BAR(B_TFULL + i), 1); mbar_init(BAR(B_TEMPTY + i), 4); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(B_QFULL + i), 1);
      mbar_init(BAR(B_QEMPTY + i), 2);     // both issuers release a Q block
      mbar_init(BAR(B_STAT + i), kEpiWarps);
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
  const float2 scale22 = make_float2(scale2, scale2);

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    int stage = 0, qb = 0;
    uint32_t phase = 0, qphase[2] = {0, 0};
    bool ok = true;
    for (int k = 0; k < a.steps && ok; ++k) {
      const Block x = block_of(a, k);
      if (!x.valid) break;
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
      if (!ok) break;
      if (elect_one()) {
        mbar_expect_tx(BAR(B_QFULL + qb), (uint32_t)lay.tile_bytes);
        for (int kb = 0; kb < KB; ++kb)
          tma_load_2d(smem_u32(sQ + (size_t)qb * lay.tile_bytes + (size_t)kb * kTile * 128), &maps.q, kb * 64,
                      x.head * a.N + x.b * kTile, BAR(B_QFULL + qb));
      }
      __syncwarp();
      qphase[qb] ^= 1;
      qb ^= 1;
      const int krow0 = x.head / a.group * a.N, T = x.b + 1;
      for (int s = 0; s < 2 * T; ++s) {
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
        if (!ok) break;
        if (elect_one()) {
          mbar_expect_tx(BAR(B_FULL + stage), (uint32_t)lay.tile_bytes);
#pragma unroll
          for (int kb = 0; kb < KB; ++kb)
            tma_load_2d(smem_u32(sK + (size_t)stage * lay.tile_bytes + (size_t)kb * kTile * 128), &maps.k, kb * 64,
                        krow0 + (s < T ? s : s - T) * kTile, BAR(B_FULL + stage));
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
    // every tcgen05.commit aimed at this CTA's barriers must have arrived before the CTA exits
    for (int i = 0; i < kStages && ok; ++i) {
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_EMPTY + stage), phase ^ 1, s_abort));
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
    for (int i = 0; i < 2 && ok; ++i, qb ^= 1)
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QEMPTY + qb), qphase[qb] ^ 1, s_abort));
  } else if (warp == 1 || warp == 6) {
    // ------------------------------------------------------------ MMA issuers.  A block is an even number of steps, so
    // step s of a block always belongs to issuer s & 1, as do its stage and its accumulator
    const int me = warp == 1 ? 0 : 1;
    int qb = 0, stage = me, acc = me;
    uint32_t sphase = 0, aphase = 0, qphase[2] = {0, 0};
    const uint32_t idesc = instr_desc(128, 128);
    const uint64_t desc_hi = smem_desc(0);
    bool ok = true;
    for (int k = 0; k < a.steps && ok; ++k) {
      const Block x = block_of(a, k);
      if (!x.valid) break;
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_QFULL + qb), qphase[qb], s_abort));
      if (!ok) break;
      qphase[qb] ^= 1;
      const uint32_t q_lo = smem_u32(sQ + (size_t)qb * lay.tile_bytes) >> 4;
      const int T = x.b + 1;
      for (int s = me; s < 2 * T; s += 2) {
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_FULL + stage), sphase, s_abort) &&
                                         mbar_wait(BAR(B_TEMPTY + acc), aphase ^ 1, s_abort));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * 128u;
        const uint32_t k_lo = smem_u32(sK + (size_t)stage * lay.tile_bytes) >> 4;
        const bool rows_first = s < T;               // first walk: D[row, key]
        if (elect_one()) {
#pragma unroll
          for (int kb = 0; kb < KB; ++kb)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const uint32_t at = (uint32_t)((kb * kTile * 128 + kk * 32) >> 4);
              const uint64_t kd = desc_hi | (uint64_t)(k_lo + at), qd = desc_hi | (uint64_t)(q_lo + at);
              if (rows_first) tc_mma(d_tmem, qd, kd, idesc, (kb | kk) ? 1u : 0u);
              else tc_mma(d_tmem, kd, qd, idesc, (kb | kk) ? 1u : 0u);
            }
          tc_commit(BAR(B_EMPTY + stage));
          tc_commit(BAR(B_TFULL + acc));
        }
        __syncwarp();
        stage += 2;
        if (stage >= kStages) { stage -= kStages; sphase ^= 1; }
        acc ^= 2;
        if (acc == me) aphase ^= 1;
      }
      if (!ok) break;
      if (elect_one()) tc_commit(BAR(B_QEMPTY + qb));
      __syncwarp();
      qb ^= 1;
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp < 6 ? warp - 2 : warp - 3;  // 0..15
    const int grp = ew >> 2;
    const int quad = warp & 3;                      // TMEM lane quadrant this warp may read
    const int row = quad * 32 + lane;               // first walk: this thread's query row; second: its key
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    float* myOff = sOff + ew * kTile;
    int n = 0;                                      // steps of this CTA so far: accumulator n & 3
    bool ok = true;
    auto done_with = [&](int acc) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TEMPTY + acc));
    };
    for (int k = 0; k < a.steps && ok; ++k) {
      const Block x = block_of(a, k);
      if (!x.valid) break;
      const int T = x.b + 1;
      // ---- first walk: the row's running max and sum over the tiles of this group
      float m_run = -INFINITY, z_run = 0.f;
      for (int t = 0; t < T; ++t, ++n) {
        if ((n & (kGroups - 1)) != grp) continue;
        const int acc = n & 3;
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_TFULL + acc), (uint32_t)((n >> 2) & 1), s_abort));
        if (!ok) break;
        tc_fence_after();
        const bool tail = t == T - 1;               // row i sees the first i + 1 keys of the block's last tile
#pragma unroll
        for (int c0 = 0; c0 < kTile; c0 += kCols) {
          uint32_t r[kCols];
          tc_ld32(lane_addr + (uint32_t)(acc * 128 + c0), r);
          tc_wait_ld();
          if (tail) {
#pragma unroll
            for (int i = 0; i < kCols; ++i)
              if (c0 + i > row) r[i] = __float_as_uint(-INFINITY);
          }
          float cm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int i = 0; i < kCols; ++i) cm4[i & 3] = fmaxf(cm4[i & 3], __uint_as_float(r[i]));
          const float cm = fmaxf(fmaxf(cm4[0], cm4[1]), fmaxf(cm4[2], cm4[3]));
          if (cm > m_run) {
            z_run *= ex2((m_run - cm) * scale2);
            m_run = cm;
          }
          if (m_run > -INFINITY) {
            const float2 ms = make_float2(-m_run * scale2, -m_run * scale2);
            float2 zs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int i = 0; i < kCols; i += 2)
              zs[(i >> 1) & 1] = __fadd2_rn(zs[(i >> 1) & 1], weight2(i, __ffma2_rn(pair_of(r, i), scale22, ms)));
            z_run += (zs[0].x + zs[0].y) + (zs[1].x + zs[1].y);
          }
        }
        done_with(acc);
      }
      if (!ok) break;
      // ---- the groups' pairs of every row -> one offset per row: max + log2(sum) + log2(128).  A query row beyond the
      // end of the sequence does not exist: an infinite offset takes it out of every column sum
      const int buf = k & 1;
      sStat[(buf * kGroups + grp) * kTile + row] = make_float2(m_run * scale2, z_run);
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_STAT + buf));
      ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_STAT + buf), (uint32_t)((k >> 1) & 1), s_abort));
      if (!ok) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = q * 32 + lane;
        float M = -INFINITY, z = 0.f;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) M = fmaxf(M, sStat[(buf * kGroups + g) * kTile + i].x);
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
          const float2 o = sStat[(buf * kGroups + g) * kTile + i];
          if (o.x > -INFINITY) z += o.y * exp2f(o.x - M);
        }
        myOff[i] = (z > 0.f && x.b * kTile + i < a.N) ? -(M + log2f(z) + 7.f) : -INFINITY;
      }
      __syncwarp();
      // ---- second walk: this thread's key, summed over the rows (of which the last block may have fewer; what stands in their
      // place is another head's query or zero, and its score at a key with an infinite element may be NaN: left out)
      const int rows_here = min(kTile, a.N - x.b * kTile);
      float* out = a.scores + (int64_t)x.head * 64 * a.nb * (a.nb + 1) + (int64_t)64 * x.b * (x.b + 1);
      for (int t = 0; t < T; ++t, ++n) {
        if ((n & (kGroups - 1)) != grp) continue;
        const int acc = n & 3;
        ok = __all_sync(0xffffffffu, mbar_wait(BAR(B_TFULL + acc), (uint32_t)((n >> 2) & 1), s_abort));
        if (!ok) break;
        tc_fence_after();
        const bool tail = t == T - 1;
        float2 cs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (!RAGGED || rows_here == kTile) {
#pragma unroll
          for (int c0 = 0; c0 < kTile; c0 += kCols) {
            uint32_t r[kCols];
            tc_ld32(lane_addr + (uint32_t)(acc * 128 + c0), r);
            tc_wait_ld();
            if (tail) {                               // key i is seen by rows i .. 127 of the block
#pragma unroll
              for (int i = 0; i < kCols; ++i)
                if (c0 + i < row) r[i] = __float_as_uint(-INFINITY);
            }
            const float4* off4 = reinterpret_cast<const float4*>(myOff + c0);
#pragma unroll
            for (int i = 0; i < kCols; i += 4) {
              const float4 off = off4[i >> 2];
              cs[0] = __fadd2_rn(cs[0], weight2(i, __ffma2_rn(pair_of(r, i), scale22, make_float2(off.x, off.y))));
              cs[1] = __fadd2_rn(cs[1], weight2(i + 2, __ffma2_rn(pair_of(r, i + 2), scale22, make_float2(off.z, off.w))));
            }
          }
        } else {
#pragma unroll
          for (int c0 = 0; c0 < kTile; c0 += kCols) {
            if (c0 >= rows_here) break;
            uint32_t r[kCols];
            tc_ld32(lane_addr + (uint32_t)(acc * 128 + c0), r);
            tc_wait_ld();
            if (tail) {
#pragma unroll
              for (int i = 0; i < kCols; ++i)
                if (c0 + i < row) r[i] = __float_as_uint(-INFINITY);
            }
            if (c0 + kCols > rows_here) {
#pragma unroll
              for (int i = 0; i < kCols; ++i)
                if (c0 + i >= rows_here) r[i] = __float_as_uint(-INFINITY);
            }
            const float4* off4 = reinterpret_cast<const float4*>(myOff + c0);
#pragma unroll
            for (int i = 0; i < kCols; i += 4) {
              const float4 off = off4[i >> 2];
              cs[0] = __fadd2_rn(cs[0], weight2(i, __ffma2_rn(pair_of(r, i), scale22, make_float2(off.x, off.y))));
              cs[1] = __fadd2_rn(cs[1], weight2(i + 2, __ffma2_rn(pair_of(r, i + 2), scale22, make_float2(off.z, off.w))));
            }
          }
        }
        out[t * kTile + row] = (cs[0].x + cs[0].y) + (cs[1].x + cs[1].y);
        done_with(acc);
      }
    }
  }

  // ---------------------------------------------------------------- teardown
  if (*s_abort)
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tc_dealloc(tmem_base, kTmemCols);
  }
  if (tid == 0 && *s_abort) set_status(a.status, TASKKV_ETIMEOUT);
}

template <int D, bool RAGGED>
cudaError_t launch_prefix_d(const void* q, const void* k, int heads, int group, int N, float* scores, int32_t* status,
                            cudaStream_t s) {
  const int n_sm = sm_count();
  const PrefixLayout lay = make_prefix_layout(D);
  cudaError_t e = cudaFuncSetAttribute(prefix_score_kernel<D, RAGGED>, cudaFuncAttributeMaxDynamicSharedMemorySize, lay.total);
  if (e != cudaSuccess) return e;
  PrefixMaps maps;
  if (!make_tensor_map_2d(&maps.k, k, D, (uint64_t)(heads / group) * (uint64_t)N, kTile)) return cudaErrorUnknown;
  if (!make_tensor_map_2d(&maps.q, q, D, (uint64_t)heads * (uint64_t)N, kTile)) return cudaErrorUnknown;
  PrefixArgs a;
  a.N = N;
  a.nb = (N + kTile - 1) / kTile;
  a.heads = heads;
  a.group = group;
  // heads whose keys take about 32 MB together: a quarter of L2, which keeps a copy on either side of the die
  int64_t kv_team = (int64_t)(32 << 20) / ((int64_t)N * D * 2);
  if (kv_team < 1) kv_team = 1;
  a.team = (int)(kv_team * group < heads ? kv_team * group : heads);
  const int64_t items = (int64_t)heads * a.nb;
  if (items > 0x3fffffff) return cudaErrorInvalidValue;
  a.items = (int)items;
  const int grid = a.items < n_sm ? a.items : n_sm;
  a.steps = (a.items + grid - 1) / grid;
  a.scores = scores;
  a.status = status;
  LaunchScope ls(K_WINDOW_TC, s);
  prefix_score_kernel<D, RAGGED><<<grid, kThreads, lay.total, s>>>(maps, a, lay);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_prefix_scores(const void* q, const void* k, int d, int heads, int group, int N, float* scores,
                                 int32_t* status, cudaStream_t s) {
  if (N % kTile)
    return d == 64 ? launch_prefix_d<64, true>(q, k, heads, group, N, scores, status, s)
                   : launch_prefix_d<128, true>(q, k, heads, group, N, scores, status, s);
  return d == 64 ? launch_prefix_d<64, false>(q, k, heads, group, N, scores, status, s)
                 : launch_prefix_d<128, false>(q, k, heads, group, N, scores, status, s);
}

}  // namespace taskkv

// Decode attention over the ragged per-head cache (Eq. 1, one query row per
// head, no mask): o_a = softmax(q_a K_u^T / sqrt(d)) V_u over the len_u rows of
// the KV head's segment, for the G query heads that share it.
//
// Split-K: a unit's rows are cut into work items of 512 rows (fewer in small caches: UnitItems), numbered once at
// compression for every unit at its capacity (so a 32768-row full head and a 772-row pruned head
// load the SMs alike; items beyond a segment's current length are skipped).  Each item produces an un-normalised partial
// (running max, sum, weighted V) per head with an online softmax in fp32; one
// combine pass merges a unit's partials.  K/V rows are read once, as 16-byte
// vectors, by all G heads.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace taskkv {

namespace {

constexpr int kAttnThreads = 128;
constexpr int kAttnWarps = kAttnThreads / 32;
constexpr int kUnroll = 4;

// PAGED (both attention kernels): the rows of a unit live in pages of the shared pool; the rows one loop iteration
// touches never cross a page (a page holds a multiple of 64 rows).  A work item's 512 rows lie in at most 8 pages:
// every lane reads one of their table entries when the item starts (lane i and i + 8, ... hold the i-th), and an
// iteration gets its page by a shuffle, so no table load sits between an iteration and its row loads.
struct ItemPages {
  int first;   // table index of the item's first page
  int mine;    // page held by this lane
};
__device__ __forceinline__ ItemPages item_pages(const DeviceProblem& p, int u, int rbeg, int lane) {
  ItemPages ip;
  ip.first = rbeg / p.page_rows;
  const int pi = ip.first + (lane & 7);
  ip.mine = pi < p.page_stride ? p.page_tab[(size_t)u * p.page_stride + pi] : 0;
  return ip;
}
// Walks the item's rows in steps of at most one page: where() gives the pool row of the current row minus that row's
// index (for all lanes of a converged warp), advance() moves on.  One division per item instead of one per step.
struct PageWalk {
  int pi;    // page of the current row, counted from the item's first
  int rem;   // its row within that page
  __device__ __forceinline__ void start(const DeviceProblem& p, const ItemPages& ip, int r) {
    pi = r / p.page_rows - ip.first;
    rem = r % p.page_rows;
  }
  __device__ __forceinline__ size_t where(const DeviceProblem& p, const ItemPages& ip, int r) const {
    const int pg = __shfl_sync(0xffffffffu, ip.mine, pi);
    return (size_t)((int64_t)pg * p.page_rows + rem - r);
  }
  __device__ __forceinline__ void advance(const DeviceProblem& p, int step) {
    rem += step;
    if (rem >= p.page_rows) {
      rem -= p.page_rows;
      ++pi;
    }
  }
};
// One work item of the scalar path: rows [rbeg, rend) of unit u for the G heads of view unit vu (row new_r, if it is
// among them, comes from kn_row / vn_row).  Leaves every row sub-group's running max, sum and weighted V in shared
// memory.  AHEAD: the next iteration's rows are requested before this one's are used, for grids that leave the SMs
// few warps; the arithmetic is the same.
template <typename T, int D, int G, bool PAGED>
struct ScalarItem {
  static constexpr int EPL = 16 / (int)sizeof(T);          // elements per lane (one 16-byte vector)
  static constexpr int LPR = D / EPL;                      // lanes per row
  static constexpr int RPW = 32 / LPR;                     // rows per warp instruction
  static constexpr int NSG = kAttnWarps * RPW;             // row sub-groups per block
  static constexpr int ROW_BYTES = D * (int)sizeof(T);
  struct Smem {
    float m[NSG][G], l[NSG][G];
    __align__(16) float acc[NSG][G][D];
  };
  template <bool AHEAD>
  __device__ __forceinline__ static void run(const DeviceProblem& p, const T* __restrict__ q, int vu, int64_t seg, int rbeg,
                                             int rend, int new_r, const unsigned char* kn_row, const unsigned char* vn_row,
                                             const ItemPages& ip, Smem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sg = lane / LPR, sl = lane % LPR;
    const int gsg = warp * RPW + sg;
    const float scale2 = kLog2e * rsqrtf((float)D);
    const unsigned char* kp = static_cast<const unsigned char*>(p.k_pool) + (PAGED ? 0 : (size_t)seg * ROW_BYTES) + sl * 16;
    const unsigned char* vp = static_cast<const unsigned char*>(p.v_pool) + (PAGED ? 0 : (size_t)seg * ROW_BYTES) + sl * 16;

    float qf[G][EPL];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint4 raw = *reinterpret_cast<const uint4*>(q + ((size_t)vu * G + g) * D + sl * EPL);
      Vec16<T>::unpack(raw, qf[g]);
#pragma unroll
      for (int e = 0; e < EPL; ++e) qf[g][e] *= scale2;
    }
    float m[G], l[G], acc[G][EPL];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      m[g] = -INFINITY;
      l[g] = 0.f;
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[g][e] = 0.f;
    }

    // two copies of the row loop: only the item that holds the new token's row pays for telling it apart
    auto rows_loop = [&](auto has_new) {
    PageWalk pw{0, 0};
    if (PAGED) pw.start(p, ip, rbeg);
    auto load = [&](int base, uint4 (&kraw)[kUnroll], uint4 (&vraw)[kUnroll]) {
      const int r0 = base + gsg;
      // pool row of row `base` minus base: adding a row index of this iteration gives its pool row
      size_t rowoff = 0;
      if (PAGED) {
        rowoff = pw.where(p, ip, base);
        pw.advance(p, NSG * kUnroll);
      }
      // one 64-bit address per array and iteration; the unrolled loads differ by compile-time offsets
      const unsigned char* kb = kp + (rowoff + (size_t)r0) * ROW_BYTES;
      const unsigned char* vb = vp + (rowoff + (size_t)r0) * ROW_BYTES;
#pragma unroll
      for (int i = 0; i < kUnroll; ++i) {
        const int r = r0 + i * NSG;
        if (r < rend) {
          kraw[i] = *reinterpret_cast<const uint4*>((decltype(has_new)::value && r == new_r) ? kn_row + sl * 16
                                                                                             : kb + i * NSG * ROW_BYTES);
          vraw[i] = *reinterpret_cast<const uint4*>((decltype(has_new)::value && r == new_r) ? vn_row + sl * 16
                                                                                             : vb + i * NSG * ROW_BYTES);
        } else {
          kraw[i] = make_uint4(0, 0, 0, 0);
          vraw[i] = make_uint4(0, 0, 0, 0);
        }
      }
    };
    auto use = [&](int base, const uint4 (&kraw)[kUnroll], const uint4 (&vraw)[kUnroll]) {
      const int r0 = base + gsg;
      float s[kUnroll][G];
#pragma unroll
      for (int i = 0; i < kUnroll; ++i) {
        float kf[EPL];
        Vec16<T>::unpack(kraw[i], kf);
#pragma unroll
        for (int g = 0; g < G; ++g) {
          float d0 = 0.f;
#pragma unroll
          for (int e = 0; e < EPL; ++e) d0 = fmaf(qf[g][e], kf[e], d0);
          s[i][g] = d0;
        }
      }
#pragma unroll
      for (int i = 0; i < kUnroll; ++i)
#pragma unroll
        for (int g = 0; g < G; ++g) {
          float v = s[i][g];
#pragma unroll
          for (int o = LPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          s[i][g] = (r0 + i * NSG < rend) ? v : -INFINITY;
        }
      float pw[kUnroll][G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        float mn = m[g];
#pragma unroll
        for (int i = 0; i < kUnroll; ++i) mn = fmaxf(mn, s[i][g]);
        const float mu = (mn == -INFINITY) ? 0.f : mn;
        const float corr = exp2f(m[g] - mu);
        float ps = 0.f;
#pragma unroll
        for (int i = 0; i < kUnroll; ++i) {
          pw[i][g] = exp2f(s[i][g] - mu);
          ps += pw[i][g];
        }
        l[g] = l[g] * corr + ps;
        m[g] = mn;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[g][e] *= corr;
      }
#pragma unroll
      for (int i = 0; i < kUnroll; ++i) {
        float vf[EPL];
        Vec16<T>::unpack(vraw[i], vf);
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
          for (int e = 0; e < EPL; ++e) acc[g][e] = fmaf(pw[i][g], vf[e], acc[g][e]);
      }
    };
    constexpr int kStep = NSG * kUnroll;
    if constexpr (AHEAD) {
      uint4 k0[kUnroll], v0[kUnroll], k1[kUnroll], v1[kUnroll];
      load(rbeg, k0, v0);
      for (int base = rbeg; base < rend; base += 2 * kStep) {     // warp-uniform trip count
        if (base + kStep < rend) load(base + kStep, k1, v1);
        use(base, k0, v0);
        if (base + 2 * kStep < rend) load(base + 2 * kStep, k0, v0);
        if (base + kStep < rend) use(base + kStep, k1, v1);
      }
    } else {
      for (int base = rbeg; base < rend; base += kStep) {         // warp-uniform trip count
        uint4 kraw[kUnroll], vraw[kUnroll];
        load(base, kraw, vraw);
        use(base, kraw, vraw);
      }
    }
    };
    if (new_r >= rbeg && new_r < rend) rows_loop(std::true_type{}); else rows_loop(std::false_type{});

#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (sl == 0) { sm.m[gsg][g] = m[g]; sm.l[gsg][g] = l[g]; }
#pragma unroll
      for (int e = 0; e < EPL; ++e) sm.acc[gsg][g][sl * EPL + e] = acc[g][e];
    }
  }
};

// ---------------------------------------------------------------------------------------------
// Grouped-query variant for bf16 (G >= 2 query heads per KV head): with several heads per row the
// scalar kernel above runs out of issue slots long before HBM, so the two contractions go through
// warp-level mma (m16n8k16, bf16 x bf16 -> fp32) on operands taken straight from 16-byte global
// loads -- no shared-memory staging; the fragment layouts are met by permuting the contraction
// index instead:
//   S^T[head, row] = Q K^T   A = Q (heads on the 16 M rows, rows >= G zero), B = 8 cache rows.  Lane
//       (g = lane/4, t = lane%4) owns cache row g and loads its 16-byte pieces i*4 + t; the two
//       halves of piece i are the lane's operand words of k-chunks 2i and 2i+1.  Q is loaded with the
//       same rule, so both sides agree on which d sits in which k slot.
//   O^T[d, head] += V^T P^T   the accumulator fragment of S^T (head g, rows 2t, 2t+1) is already the
//       B fragment of P^T; the A fragment needs pairs of consecutive rows at one d, built with one
//       byte-permute from the lane's loads of rows 2t, 2t+1, 2t+8, 2t+9 (piece g of each 128-byte
//       line).  Accumulator row (m-block mb, half hf) of lane g stands for d = pd(mb, hf, g).
// P is rounded to bf16 for the second product (fp32 accumulation); the normaliser is summed in fp32.
// Each warp walks 16-row blocks of the work item with its own running (max, sum, O^T); the four
// warps are merged like the sub-groups of the scalar kernel and the partial goes to the same slots.
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// One work item of the warp-mma path (see ScalarItem): the sub-groups are the block's four warps.
template <int D, int G, bool PAGED>
struct MmaItem {
  static constexpr int NSG = kAttnWarps;
  static constexpr int ROW_BYTES = D * 2;
  static constexpr int KC = D / 16;            // k-chunks of the first product
  static constexpr int KP = D / 32;            // 16-byte pieces of a K row per lane
  static constexpr int MB = D / 16;            // m-blocks (16 d each) of the second product
  static constexpr int VP = D / 64;            // 16-byte pieces of a V row per lane
  static constexpr int kBlk = 16;              // cache rows per warp iteration
  struct Smem {
    float m[NSG][G], l[NSG][G];
    __align__(16) float acc[NSG][G][D];
  };
  template <bool AHEAD>
  __device__ __forceinline__ static void run(const DeviceProblem& p, const __nv_bfloat16* __restrict__ q, int vu, int64_t seg,
                                             int rbeg, int rend, int new_r, const unsigned char* kn_row,
                                             const unsigned char* vn_row, const ItemPages& ip, Smem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const float scale2 = kLog2e * rsqrtf((float)D);
    // d of accumulator row (mb, hf) of this lane's two output rows: e = hf * MB + mb, piece e / 8, element e % 8
    auto pd = [&](int mb, int hf, int gg) { const int e = hf * MB + mb; return (e >> 3) * 64 + gg * 8 + (e & 7); };
    const unsigned char* kp = static_cast<const unsigned char*>(p.k_pool);
    const unsigned char* vp = static_cast<const unsigned char*>(p.v_pool);

    // Q fragments: head g on M row g
    uint32_t qa[KC][2];
#pragma unroll
    for (int i = 0; i < KP; ++i) {
      uint4 raw = make_uint4(0, 0, 0, 0);
      if (g < G) raw = *reinterpret_cast<const uint4*>(q + ((size_t)vu * G + g) * D + (i * 4 + t) * 8);
      qa[2 * i][0] = raw.x; qa[2 * i][1] = raw.y;
      qa[2 * i + 1][0] = raw.z; qa[2 * i + 1][1] = raw.w;
    }
    float m_run = -INFINITY, l_run = 0.f;   // head g (this lane's share of the sum)
    float o[MB][4];
#pragma unroll
    for (int mb = 0; mb < MB; ++mb)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[mb][e] = 0.f;

    // byte offset of this lane's first K vector (row g, piece t) and V vector (row 2t, piece g) within a block
    const int klane = g * ROW_BYTES + t * 16, vlane = 2 * t * ROW_BYTES + g * 16;
    // two copies of the row loop: only the item that holds the new token's row pays for telling it apart
    auto rows_loop = [&](auto has_new) {
    PageWalk pw{0, 0};
    if (PAGED) pw.start(p, ip, rbeg + warp * kBlk);
    // kb, vb: this lane's first K and V vector of the next 16-row block to load; the unrolled loads differ from them by
    // compile-time offsets.  Contiguous layout: row r of the unit is pool row seg + r, the pointers step from block
    // to block; paged: they are set from the block's page.
    const unsigned char* kb = kp + ((size_t)seg + (size_t)(rbeg + warp * kBlk)) * ROW_BYTES + klane;
    const unsigned char* vb = vp + ((size_t)seg + (size_t)(rbeg + warp * kBlk)) * ROW_BYTES + vlane;
    auto load = [&](int blk, uint4 (&kraw)[2][KP], uint4 (&vraw)[4][VP]) {
      if (PAGED) {
        // pool row of row `blk` minus blk: adding a row index of this 16-row block gives its pool row
        const size_t rowoff = pw.where(p, ip, blk);
        pw.advance(p, kAttnWarps * kBlk);
        kb = kp + (rowoff + (size_t)blk) * ROW_BYTES + klane;
        vb = vp + (rowoff + (size_t)blk) * ROW_BYTES + vlane;
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = blk + 8 * j + g;
#pragma unroll
        for (int i = 0; i < KP; ++i)
          kraw[j][i] = r < rend ? *reinterpret_cast<const uint4*>((decltype(has_new)::value && r == new_r)
                                                                      ? kn_row + (i * 4 + t) * 16
                                                                      : kb + j * 8 * ROW_BYTES + i * 64)
                                : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int r = blk + 2 * t + (x & 1) + 8 * (x >> 1);
#pragma unroll
        for (int i = 0; i < VP; ++i)
          vraw[x][i] = r < rend ? *reinterpret_cast<const uint4*>((decltype(has_new)::value && r == new_r)
                                                                      ? vn_row + i * 128 + g * 16
                                                                      : vb + ((x & 1) + 8 * (x >> 1)) * ROW_BYTES + i * 128)
                                : make_uint4(0, 0, 0, 0);
      }
      if (!PAGED) {
        kb += kAttnWarps * kBlk * ROW_BYTES;
        vb += kAttnWarps * kBlk * ROW_BYTES;
      }
    };
    auto use = [&](int blk, const uint4 (&kraw)[2][KP], const uint4 (&vraw)[4][VP]) {
      // S^T for the two 8-row halves of the block
      float sc[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int e = 0; e < 4; ++e) sc[j][e] = 0.f;
#pragma unroll
        for (int i = 0; i < KP; ++i) {
          mma_bf16_16816(sc[j], qa[2 * i][0], 0u, qa[2 * i][1], 0u, kraw[j][i].x, kraw[j][i].y);
          mma_bf16_16816(sc[j], qa[2 * i + 1][0], 0u, qa[2 * i + 1][1], 0u, kraw[j][i].z, kraw[j][i].w);
        }
      }
      // online softmax for head g over rows blk + 8j + 2t + {0, 1}
      float tv[4];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int r = blk + 8 * j + 2 * t + e;
          tv[2 * j + e] = r < rend ? sc[j][e] * scale2 : -INFINITY;
        }
      float mx = fmaxf(fmaxf(tv[0], tv[1]), fmaxf(tv[2], tv[3]));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float mn = fmaxf(m_run, mx);
      const float mu = (mn == -INFINITY) ? 0.f : mn;
      const float corr = exp2f(m_run - mu);
      float pw[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) pw[e] = exp2f(tv[e] - mu);
      l_run = l_run * corr + ((pw[0] + pw[1]) + (pw[2] + pw[3]));
      m_run = mn;
      // rescale O^T: its columns are heads 2t, 2t+1, whose factors live in lanes 8t and 8t + 4
      const float ca = __shfl_sync(0xffffffffu, corr, 8 * t);
      const float cb = __shfl_sync(0xffffffffu, corr, 8 * t + 4);
      if (__any_sync(0xffffffffu, corr != 1.f)) {
#pragma unroll
        for (int mb = 0; mb < MB; ++mb) {
          o[mb][0] *= ca; o[mb][1] *= cb; o[mb][2] *= ca; o[mb][3] *= cb;
        }
      }
      const uint32_t pb0 = pack_bf16(pw[0], pw[1]);   // rows 2t, 2t+1
      const uint32_t pb1 = pack_bf16(pw[2], pw[3]);   // rows 2t+8, 2t+9
#pragma unroll
      for (int mb = 0; mb < MB; ++mb) {
        uint32_t a[4];
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int e = hf * MB + mb, pc = e >> 3, wi = (e & 7) >> 1;
          const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
          a[hf] = __byte_perm(word_of(vraw[0][pc], wi), word_of(vraw[1][pc], wi), sel);       // rows 2t, 2t+1
          a[2 + hf] = __byte_perm(word_of(vraw[2][pc], wi), word_of(vraw[3][pc], wi), sel);   // rows 2t+8, 2t+9
        }
        mma_bf16_16816(o[mb], a[0], a[1], a[2], a[3], pb0, pb1);
      }
    };
    constexpr int kStep = kAttnWarps * kBlk;
    const int first = rbeg + warp * kBlk;
    if constexpr (AHEAD) {
      uint4 k0[2][KP], v0[4][VP], k1[2][KP], v1[4][VP];
      if (first < rend) load(first, k0, v0);
      for (int blk = first; blk < rend; blk += 2 * kStep) {       // warp-uniform
        if (blk + kStep < rend) load(blk + kStep, k1, v1);
        use(blk, k0, v0);
        if (blk + 2 * kStep < rend) load(blk + 2 * kStep, k0, v0);
        if (blk + kStep < rend) use(blk + kStep, k1, v1);
      }
    } else {
      for (int blk = first; blk < rend; blk += kStep) {           // warp-uniform
        uint4 kraw[2][KP], vraw[4][VP];
        load(blk, kraw, vraw);
        use(blk, kraw, vraw);
      }
    }
    };
    if (new_r >= rbeg && new_r < rend) rows_loop(std::true_type{}); else rows_loop(std::false_type{});

    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    if (t == 0 && g < G) { sm.m[warp][g] = m_run; sm.l[warp][g] = l_run; }
#pragma unroll
    for (int mb = 0; mb < MB; ++mb)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int head = 2 * t + (e & 1);
        if (head < G) sm.acc[warp][head][pd(mb, e >> 1, g)] = o[mb][e];
      }
  }
};

// Work items that hold the first `len` rows of a unit.  (Where the reserve is cut like the rest, the usual case, its first
// row does not matter and the unit's capacity is not read.)
template <bool TAIL>
__device__ __forceinline__ int unit_item_count(const DeviceProblem& p, int unit, int len) {
  if (!TAIL || p.dec_tail == p.dec_shift) return (len + p.dec_chunk - 1) >> p.dec_shift;
  return UnitItems<>(p.cap[unit] - p.max_new, p.dec_shift, p.dec_tail).count(len);
}

template <typename T, int D, int G, bool PAGED>
using Item = typename std::conditional<sizeof(T) == 2, MmaItem<D, G, PAGED>, ScalarItem<T, D, G, PAGED>>::type;

// Merges the sub-groups an item left in shared memory: emit(head, d, weighted V, max, sum) for this thread's elements.
template <int NSG, int D, int G, class Smem, class Emit>
__device__ __forceinline__ void merge_item(const Smem& sm, const Emit& emit) {
  for (int i = threadIdx.x; i < G * D; i += kAttnThreads) {
    const int hh = i / D, dd = i % D;
    float M = -INFINITY;
#pragma unroll
    for (int x = 0; x < NSG; ++x) M = fmaxf(M, sm.m[x][hh]);
    float a = 0.f, ll = 0.f;
#pragma unroll
    for (int x = 0; x < NSG; ++x) {
      const float mx = sm.m[x][hh];
      const float w = (mx == -INFINITY) ? 0.f : exp2f(mx - M);
      a = fmaf(w, sm.acc[x][hh][dd], a);
      ll = fmaf(w, sm.l[x][hh], ll);
    }
    emit(hh, dd, a, M, ll);
  }
}

// The new token's K and V rows into the segment of unit u at row new_r, by the block whose work item holds that row
// (only it touches the unit's new row).  s_word: a shared word free for use here.
template <int ROW_BYTES, bool PAGED>
__device__ __forceinline__ void store_new_row(const DeviceProblem& p, int u, int64_t seg, int new_r,
                                              const unsigned char* kn_row, const unsigned char* vn_row, int* s_word) {
  const int tid = threadIdx.x;
  bool have_page = true;
  if (PAGED && new_r % p.page_rows == 0) {
    // the appended row opens a new page: one comes off the pool
    if (tid == 0) {
      const int at = pool_pop(p, 1);
      if (at >= 0) p.page_tab[(size_t)u * p.page_stride + new_r / p.page_rows] = p.pool_free[at];
      *s_word = at;
    }
    __syncthreads();
    have_page = *s_word >= 0;                       // an empty pool: status ESTATE, the row is not stored
  }
  if (have_page && tid < ROW_BYTES / 16) {
    const size_t drow = pool_row(p, u, seg, new_r);
    unsigned char* kd = static_cast<unsigned char*>(p.k_pool) + drow * ROW_BYTES + tid * 16;
    unsigned char* vd = static_cast<unsigned char*>(p.v_pool) + drow * ROW_BYTES + tid * 16;
    *reinterpret_cast<uint4*>(kd) = *reinterpret_cast<const uint4*>(kn_row + tid * 16);
    *reinterpret_cast<uint4*>(vd) = *reinterpret_cast<const uint4*>(vn_row + tid * 16);
  }
}

template <typename T, int D, int G, bool PAGED>
__global__ void __launch_bounds__(kAttnThreads, sizeof(T) == 2 ? 4 : 1)
decode_attn_kernel(DeviceProblem p, const T* __restrict__ q, const int32_t* __restrict__ lengths,
                   const unsigned char* __restrict__ k_new, const unsigned char* __restrict__ v_new, T* __restrict__ out,
                   int early) {
  using It = Item<T, D, G, PAGED>;
  constexpr int ROW_BYTES = It::ROW_BYTES;
  __shared__ typename It::Smem sm;
  __shared__ int s_word;
  __shared__ int s_direct;     // >= 0: the item is its unit's only one, the output goes to view unit s_direct

  const int tid = threadIdx.x, lane = tid & 31;
  // The table of work items is written when the cache is planned, not by the kernel before this one in the
  // stream: the block's first entry is read before the wait, under that kernel's tail.  (With a search of the units'
  // offsets in its place 384 units of 1500 to 6000 rows took 60.9 us instead of 59.4, 1024 units of 32768 rows 473 and 470.)
  const int item_first = p.item0 + (int)blockIdx.x;
  const int2 at_first = item_first < p.item1 ? p.dec_item[item_first] : make_int2(0, 0);
  // `early` (set by the host when the kernel before this one in the stream cannot be one that writes these units'
  // lengths or page tables: see launch_decode): the first item's unit data is read before the wait as well, and the
  // wait comes just before the block first touches what the caller's kernels produce (q, the new token's rows) or
  // writes anything.  A block none of whose items holds rows waits before it leaves: were that so for the whole grid, the
  // merge, which waits for this grid alone, and whatever follows it could overtake the kernels before this one.
  bool waited = false;
  auto wait_once = [&]() {
    if (!waited) {
      grid_dependency_wait();
      grid_launch_dependents();
      waited = true;
    }
  };
  if (!early) wait_once();
  for (int item = item_first; item < p.item1; item += gridDim.x) {
    __syncthreads();                                // previous item's shared state consumed
    const int2 at = item == item_first ? at_first : p.dec_item[item];
    if (at.x == 0) continue;                        // an item of a layer that is not in yet
    const int w = at.x - 1, rbeg = at.y & ~63;
    const LmUnit lu = lm_unit(p, w);
    const int vu = lu.v;                            // view unit: index into q and lengths
    const int u = lu.u;                             // unit: index into the cache
    int len = p.len[u];
    // fused step: the new token's row sits at index len; it is read from k_new / v_new and the item that holds
    // it also stores it in the segment (the length itself is raised by the combine pass)
    const int new_r = (k_new != nullptr && len < p.cap[u]) ? len : -1;
    if (new_r >= 0) ++len;
    if (lengths) len = min(max(lengths[vu], 0), len);
    if (rbeg >= len) continue;                      // an item of the reserve beyond the segment's length
    const int rend = min(len, rbeg + (1 << (at.y & 63)));
    if (tid == 0) s_direct = len <= p.dec_chunk ? vu : -1;     // read back after the row loop (no register held)
    const int64_t seg = p.seg_off[u];
    const unsigned char* kn_row = k_new + (size_t)vu * ROW_BYTES;
    const unsigned char* vn_row = v_new + (size_t)vu * ROW_BYTES;
    wait_once();
    if (new_r >= rbeg && new_r < rend) store_new_row<ROW_BYTES, PAGED>(p, u, seg, new_r, kn_row, vn_row, &s_word);
    ItemPages ip{0, 0};
    if (PAGED) ip = item_pages(p, u, rbeg, lane);
    It::template run<false>(p, q, vu, seg, rbeg, rend, new_r, kn_row, vn_row, ip, sm);
    __syncthreads();
    merge_item<It::NSG, D, G>(sm, [&](int hh, int dd, float a, float M, float ll) {
      if (s_direct >= 0) {
        // the unit's only item: this is Eq. 1 over the whole segment (what the combine pass would make of one
        // partial, bit for bit); the combine pass skips such units
        store_out(out + ((size_t)s_direct * G + hh) * D + dd, ll > 0.f ? a / ll : 0.f);
        return;
      }
      p.part_acc[((size_t)item * G + hh) * D + dd] = a;
      if (dd == 0) {
        p.part_ml[((size_t)item * G + hh) * 2 + 0] = M;
        p.part_ml[((size_t)item * G + hh) * 2 + 1] = ll;
      }
    });
  }
  wait_once();
}

// One block per (view unit, query head of the group): merge the unit's partials.  First the block finds
// the largest running maximum, then each warp accumulates every fourth partial against it (independent
// loads, fixed order), and the four warps are summed in shared memory.
constexpr int kCombineThreads = 256;
constexpr int kCombineWarps = kCombineThreads / 32;
constexpr int kCombineStage = 1024;     // partial results weighted per round (one round up to 524288 rows)

// One block per (view unit, query head of the group).  The weights exp2(m_i - M) of the unit's partial results
// are computed once, by all threads, into shared memory; the accumulation loop then has nothing but independent
// 16-byte loads in it (a long unit has over a hundred partials and one block: its latency is the kernel's).
// PRE: partial outputs a warp loads ahead of the weights (8: 64 registers, four blocks per SM (the lean one: six), for grids that are
// resident at once anyway -- it takes two round trips to L2 off the merge; 0: the lean variant for many thousands of
// blocks, most of them with nothing to merge).  TAIL: the reserve's items are larger than the others (a template argument,
// since a branch here costs a single layer's merge 0.2 to 0.4 us: 9.1 -> 9.5 for 8 units of up to 8000 rows).
template <typename T, int D, int G, int PRE, bool TAIL>
__global__ void __launch_bounds__(kCombineThreads, PRE > 0 ? 4 : 6) decode_combine_kernel(DeviceProblem p,
                                                                         const int32_t* __restrict__ lengths,
                                                                         int fused_step, T* __restrict__ out) {
  constexpr int EPL = D / 32;
  __shared__ float s_red[kCombineWarps];
  __shared__ float s_l[kCombineWarps];
  __shared__ float s_w[kCombineStage];
  __shared__ __align__(16) float s_acc[kCombineWarps][D];
  // Lengths, capacities and the item table are not written by the attention kernel before this one: they are read
  // before the wait, under that kernel's tail (the lengths were last written by this kernel's previous launch or by
  // an append, both complete before the attention kernel let this one start).
  const int u = blockIdx.x / G, g = blockIdx.x % G;     // u: view unit
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = view_unit(p, u);
  int len = p.len[unit];
  const bool grown = fused_step && len < p.cap[unit];   // the attention pass appends the new token's row
  const int len_next = len + (grown ? 1 : 0);
  len = len_next;
  if (lengths) len = min(max(lengths[u], 0), len);
  // the unit's items that hold rows (the table also numbers the reserve for appended tokens)
  const int i0 = p.dec_off[lm_index(p, unit)], i1 = i0 + unit_item_count<TAIL>(p, unit, len);
  grid_dependency_wait();
  grid_launch_dependents();
  if (i1 - i0 != 1) {                                   // a unit of one item has its output from the attention kernel
  const float2* ml = reinterpret_cast<const float2*>(p.part_ml);
  const int n = i1 - i0;
  // Issued together, right after the wait: this thread's (max, sum) pair and this warp's first kPre partial outputs
  // (they do not depend on the weights), so that the merge costs two round trips to L2 instead of four.
  constexpr int kPre = PRE;
  using Vec = typename std::conditional<EPL == 4, float4, float2>::type;
  Vec pre[kPre > 0 ? kPre : 1];
#pragma unroll
  for (int q = 0; q < kPre; ++q) {
    const int j = warp + q * kCombineWarps;
    if (j < n) pre[q] = *reinterpret_cast<const Vec*>(p.part_acc + ((size_t)(i0 + j) * G + g) * D + lane * EPL);
  }
  const float2 v0 = tid < n ? ml[(size_t)(i0 + tid) * G + g] : make_float2(-INFINITY, 0.f);
  float M = v0.x;
  for (int i = i0 + tid + kCombineThreads; i < i1; i += kCombineThreads) M = fmaxf(M, ml[(size_t)i * G + g].x);
  M = warp_max(M);
  if (lane == 0) s_red[warp] = M;
  __syncthreads();
  M = s_red[0];
#pragma unroll
  for (int w = 1; w < kCombineWarps; ++w) M = fmaxf(M, s_red[w]);
  float acc[EPL];
#pragma unroll
  for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
  float L = 0.f;
  auto add = [&](float wgt, const Vec& t) {
    if constexpr (EPL == 4) {
      acc[0] = fmaf(wgt, t.x, acc[0]); acc[1] = fmaf(wgt, t.y, acc[1]);
      acc[2] = fmaf(wgt, t.z, acc[2]); acc[3] = fmaf(wgt, t.w, acc[3]);
    } else {
      acc[0] = fmaf(wgt, t.x, acc[0]); acc[1] = fmaf(wgt, t.y, acc[1]);
    }
  };
  for (int c0 = i0; c0 < i1; c0 += kCombineStage) {
    const int cn = min(kCombineStage, i1 - c0);
    __syncthreads();                                    // the previous round's weights have been used
    for (int j = tid; j < cn; j += kCombineThreads) {
      const float2 v = (c0 == i0 && j == tid) ? v0 : ml[(size_t)(c0 + j) * G + g];
      const float wgt = (v.x == -INFINITY) ? 0.f : exp2f(v.x - M);
      s_w[j] = wgt;
      L = fmaf(wgt, v.y, L);
    }
    __syncthreads();
    int j = warp;                                       // every warp adds its partials in ascending order
    if (c0 == i0) {
#pragma unroll
      for (int q = 0; q < kPre; ++q, j += kCombineWarps)
        if (j < cn) add(s_w[j], pre[q]);
    }
#pragma unroll 8
    for (; j < cn; j += kCombineWarps)
      add(s_w[j], *reinterpret_cast<const Vec*>(p.part_acc + ((size_t)(c0 + j) * G + g) * D + lane * EPL));
  }
  L = warp_sum(L);
#pragma unroll
  for (int e = 0; e < EPL; ++e) s_acc[warp][lane * EPL + e] = acc[e];
  if (lane == 0) s_l[warp] = L;
  __syncthreads();
  if (tid < D) {
    float Lt = 0.f, a = 0.f;
#pragma unroll
    for (int w = 0; w < kCombineWarps; ++w) {
      Lt += s_l[w];
      a += s_acc[w][tid];
    }
    store_out(out + ((size_t)u * G + g) * D + tid, Lt > 0.f ? a / Lt : 0.f);
  }
  }
  // fused step: the last of the unit's G blocks (each has read the old length by now) raises the length
  if (fused_step && tid == 0) {
    if (atomicAdd(&p.step_cnt[unit], 1) == G - 1) {
      p.step_cnt[unit] = 0;
      // (a recorded device error -- a paged cache whose pool ran dry under this very step -- freezes the lengths:
      // no row is counted whose page may not exist)
      if (grown) { if (p.page_rows == 0 || *p.status == 0) p.len[unit] = len_next; }
      else set_status(p.status, TASKKV_ESTATE);
    }
  }
}

// Asks for rows [r0, r1) of a work item (K by warp 0, V by warp 1) to be brought into L2.  A hint only: nothing is
// ordered by it, and it may be given before the rows' writers are known to be complete.
template <int ROW_BYTES, bool PAGED>
__device__ __forceinline__ void prefetch_item(const DeviceProblem& p, const ItemPages& ip, int64_t seg, int r0, int r1) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp > 1) return;
  const unsigned char* pool = static_cast<const unsigned char*>(warp == 0 ? p.k_pool : p.v_pool);
  size_t row = (size_t)seg + (size_t)r0;
  if (PAGED) {
    const int pg = ip.first + lane;                        // lanes 0..7: one page each
    r0 = max(r0, pg * p.page_rows);
    r1 = lane < 8 ? min(r1, (pg + 1) * p.page_rows) : r0;
    row = (size_t)ip.mine * p.page_rows + (size_t)(r0 - pg * p.page_rows);
  } else if (lane > 0) {
    return;
  }
  if (r1 > r0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(pool + row * ROW_BYTES), "r"((r1 - r0) * ROW_BYTES)
                 : "memory");
}

// The merge for calls whose units have at most 32 partial results each: a warp per (view unit, query head), eight to a
// block, one partial's (max, sum) per lane and no block barrier.  The sums are formed in the order of the kernel above
// (its warp w adds partials w, w + 8, ...), so the results are the same bits.  Where units are short the block per head
// of that kernel is launch and barriers: 384 units x 4 heads of at most 12 partials, the step 65.7 -> 61.0 us; a single
// layer of units of 25 partials, three rounds for a warp, is 0.3 us slower than with a block per head.
template <typename T, int D, int G>
__global__ void __launch_bounds__(kCombineThreads) decode_combine_few_kernel(DeviceProblem p,
                                                                             const int32_t* __restrict__ lengths,
                                                                             int fused_step, T* __restrict__ out) {
  constexpr int EPL = D / 32;
  using Vec = typename std::conditional<EPL == 4, float4, float2>::type;
  const int lane = threadIdx.x & 31;
  const int vg = (int)blockIdx.x * kCombineWarps + (threadIdx.x >> 5);
  const bool there = vg < p.view_U * G;
  const int u = there ? vg / G : 0, g = vg % G;         // u: view unit
  const int unit = view_unit(p, u);
  // read before the wait, as in the kernel above
  int len = p.len[unit];
  const bool grown = fused_step && len < p.cap[unit];
  const int len_next = len + (grown ? 1 : 0);
  len = len_next;
  if (lengths) len = min(max(lengths[u], 0), len);
  const int i0 = p.dec_off[lm_index(p, unit)], n = unit_item_count<true>(p, unit, len);
  grid_dependency_wait();
  grid_launch_dependents();
  if (!there) return;
  if (n != 1) {                                         // a unit of one item has its output from the attention kernel
    const float2 v = lane < n ? reinterpret_cast<const float2*>(p.part_ml)[(size_t)(i0 + lane) * G + g]
                              : make_float2(-INFINITY, 0.f);
    const float* src = p.part_acc + ((size_t)i0 * G + g) * D + lane * EPL;
    Vec first[kCombineWarps];                           // requested together with the pairs
#pragma unroll
    for (int j = 0; j < kCombineWarps; ++j)
      if (j < n) first[j] = *reinterpret_cast<const Vec*>(src + (size_t)j * G * D);
    const float M = warp_max(v.x);
    const float w = (v.x == -INFINITY) ? 0.f : exp2f(v.x - M);
    const float L = warp_sum(fmaf(w, v.y, 0.f));
    float acc[kCombineWarps][EPL];
    auto add = [&](float (&a)[EPL], float wgt, const Vec& t) {
      a[0] = fmaf(wgt, t.x, a[0]);
      a[1] = fmaf(wgt, t.y, a[1]);
      if constexpr (EPL == 4) {
        a[2] = fmaf(wgt, t.z, a[2]);
        a[3] = fmaf(wgt, t.w, a[3]);
      }
    };
#pragma unroll
    for (int j = 0; j < kCombineWarps; ++j) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[j][e] = 0.f;
      const float wj = __shfl_sync(0xffffffffu, w, j);
      if (j < n) add(acc[j], wj, first[j]);
    }
    for (int j0 = kCombineWarps; j0 < n; j0 += kCombineWarps) {
      Vec t[kCombineWarps];
#pragma unroll
      for (int j = 0; j < kCombineWarps; ++j)
        if (j0 + j < n) t[j] = *reinterpret_cast<const Vec*>(src + (size_t)(j0 + j) * G * D);
#pragma unroll
      for (int j = 0; j < kCombineWarps; ++j) {
        const float wj = __shfl_sync(0xffffffffu, w, j0 + j);
        if (j0 + j < n) add(acc[j], wj, t[j]);
      }
    }
    T* o = out + ((size_t)u * G + g) * D + lane * EPL;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      float a = 0.f;
#pragma unroll
      for (int j = 0; j < kCombineWarps; ++j) a += acc[j][e];
      store_out(o + e, L > 0.f ? a / L : 0.f);
    }
  }
  if (fused_step && lane == 0) {
    // the last of the unit's G warps raises the length, as above
    if (atomicAdd(&p.step_cnt[unit], 1) == G - 1) {
      p.step_cnt[unit] = 0;
      if (grown) { if (p.page_rows == 0 || *p.status == 0) p.len[unit] = len_next; }
      else set_status(p.status, TASKKV_ESTATE);
    }
  }
}

// The whole of a small call in one launch: a thread-block cluster of cs CTAs owns a unit, its CTAs take the unit's work
// items (rank, rank + cs), push their partial results into the cluster's shared memory, and every CTA merges its share
// of the outputs after one cluster barrier.  The items, their arithmetic and the order in which they are merged are
// those of the two kernels above, so the results are theirs bit for bit.
// Bound by latency (a layer of a 4096-token, 32-head prompt holds 21 MB, 3.2 us of HBM time; two launches 17.2 us, this
// one 13.9; one fp32 layer of 8 heads x 512 rows 16.6 and 6.4 us, there with items of 64 rows instead of 512): it saves the second launch, the
// trip of the partial results through L2 and the search for the block's work item; an item's rows are requested into
// L2 as a whole when it starts, and where the registers allow it (d = 64, fp32) the warps, few to an SM here, load the
// next rows before they use the present ones.
constexpr int kClusterSlots = 2;         // items per CTA
constexpr int kClusterMax = 16;          // CTAs per cluster
constexpr int kClusterItems = kClusterSlots * kClusterMax;
static_assert(kClusterItems == kDecodeFewItems, "one lane per item in the merge");

template <typename T, int D, int G, bool PAGED>
__global__ void __launch_bounds__(kAttnThreads, 2)
decode_cluster_kernel(DeviceProblem p, const T* __restrict__ q, const int32_t* __restrict__ lengths,
                      const unsigned char* __restrict__ k_new, const unsigned char* __restrict__ v_new,
                      T* __restrict__ out, int early) {
  using It = Item<T, D, G, PAGED>;
  constexpr int ROW_BYTES = It::ROW_BYTES;
  constexpr bool kAhead = sizeof(T) == 4 || D == 64;
  __shared__ typename It::Smem sm;
  __shared__ float s_part[kClusterSlots * G * D];        // [item][this CTA's share of the G * D outputs]
  __shared__ float2 s_ml[G][kClusterItems];              // (max, sum) of every item
  __shared__ float s_w[G][kClusterItems], s_L[G];
  __shared__ int s_word;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int v = (int)blockIdx.x / cs, u = view_unit(p, v);
  const int share = G * D / cs;
  cl.sync();                                             // every CTA is there before anything is pushed to it
  if (!early) { grid_dependency_wait(); grid_launch_dependents(); }
  int len = p.len[u];
  const bool fused = k_new != nullptr;
  const bool grown = fused && len < p.cap[u];
  const int len_next = len + (grown ? 1 : 0), new_r = grown ? len : -1;
  const int64_t seg = p.seg_off[u];
  len = len_next;
  if (lengths) len = min(max(lengths[v], 0), len);
  const int n = (len + p.dec_chunk - 1) >> p.dec_shift;
  const int old_len = new_r >= 0 ? min(len, new_r) : len;   // rows that are in the segment already
  if (!PAGED) prefetch_item<ROW_BYTES, PAGED>(p, ItemPages{0, 0}, seg, rank * p.dec_chunk, min(old_len, (rank + 1) * p.dec_chunk));
  if (early) { grid_dependency_wait(); grid_launch_dependents(); }
  for (int j = rank; j < n; j += cs) {
    const int rbeg = j * p.dec_chunk, rend = min(len, rbeg + p.dec_chunk);
    const unsigned char* kn_row = k_new + (size_t)v * ROW_BYTES;
    const unsigned char* vn_row = v_new + (size_t)v * ROW_BYTES;
    if (new_r >= rbeg && new_r < rend) store_new_row<ROW_BYTES, PAGED>(p, u, seg, new_r, kn_row, vn_row, &s_word);
    ItemPages ip{0, 0};
    if (PAGED) {
      ip = item_pages(p, u, rbeg, lane);
      prefetch_item<ROW_BYTES, PAGED>(p, ip, seg, rbeg, min(rend, old_len));
    }
    __syncthreads();                                     // the previous item's sub-groups have been merged
    It::template run<kAhead>(p, q, v, seg, rbeg, rend, new_r, kn_row, vn_row, ip, sm);
    __syncthreads();
    merge_item<It::NSG, D, G>(sm, [&](int hh, int dd, float a, float M, float ll) {
      if (n == 1) {
        store_out(out + ((size_t)v * G + hh) * D + dd, ll > 0.f ? a / ll : 0.f);
        return;
      }
      const int i = hh * D + dd, owner = i / share;
      *cl.map_shared_rank(&s_part[j * share + (i - owner * share)], owner) = a;
      if (dd < cs) *cl.map_shared_rank(&s_ml[hh][j], dd) = make_float2(M, ll);
    });
  }
  cl.sync();                                             // all items are in; every CTA has read the length
  if (n != 1) {
    for (int hh = warp; hh < G; hh += kAttnWarps) {
      const float2 o = lane < n ? s_ml[hh][lane] : make_float2(-INFINITY, 0.f);
      const float M = warp_max(o.x);
      const float w = (o.x == -INFINITY) ? 0.f : exp2f(o.x - M);
      s_w[hh][lane] = w;
      const float L = warp_sum(fmaf(w, o.y, 0.f));
      if (lane == 0) s_L[hh] = L;
    }
    __syncthreads();
    for (int i = tid; i < share; i += kAttnThreads) {
      const int hh = (rank * share + i) / D;
      float a = 0.f;
      for (int w = 0; w < kCombineWarps; ++w) {          // the order of the combine kernel's warps
        float acc = 0.f;
        for (int j = w; j < n; j += kCombineWarps) acc = fmaf(s_w[hh][j], s_part[j * share + i], acc);
        a += acc;
      }
      const float L = s_L[hh];
      store_out(out + (size_t)v * G * D + rank * share + i, L > 0.f ? a / L : 0.f);
    }
  }
  if (fused && rank == 0 && tid == 0) {
    // (a recorded device error freezes the lengths of a paged cache, as in the combine kernel)
    if (!grown) set_status(p.status, TASKKV_ESTATE);
    else if (!PAGED || *reinterpret_cast<volatile int32_t*>(p.status) == 0) p.len[u] = len_next;
  }
}

// Whether the device co-schedules a cluster of 16 CTAs of this kernel (above the portable size, which the kernel's
// attribute allows on the devices where it was set).
template <typename T, int D, int G, bool PAGED>
bool cluster16_fits() {
  static PerDevice<> known;
  return known.get(current_device(), 0, [] {
    if (cudaFuncSetAttribute(decode_cluster_kernel<T, D, G, PAGED>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
        cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kClusterMax, 1, 1);
    cfg.blockDim = dim3(kAttnThreads, 1, 1);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kClusterMax;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, decode_cluster_kernel<T, D, G, PAGED>, &cfg) != cudaSuccess) n = 0;
    cudaGetLastError();
    return n > 0 ? 1 : 0;
  }) > 0;
}

// CTAs per unit for the one-launch form, 0 if the call is not small enough for it or its items are not all of one size (a
// reserve that is cut into longer ones is more than 32 items a unit where this form would be the faster one).  A unit gets a
// CTA per item of the longest prompt (the tokens appended since may give a CTA a second one), and all CTAs of the call
// fit on the GPU together, two to an SM: beyond that the call is bound by HBM, and the persistent attention kernel with
// its deal of equal items is the better one.
int cluster_size(const DeviceProblem& p) {
  if (p.items_cap > kClusterItems || p.dec_tail != p.dec_shift) return 0;
  int cs = 1;
  while (cs < p.items_kept || kClusterSlots * cs < p.items_cap) cs *= 2;
  if (cs > kClusterMax || (int64_t)p.view_U * cs > 2 * kSms) return 0;
  return cs;
}

template <typename T, int D, int G, bool PAGED>
cudaError_t launch_cluster(const DeviceProblem& p, int cs, const T* q, const int32_t* lengths, const unsigned char* kn,
                           const unsigned char* vn, T* out, cudaStream_t s, int early) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.view_U * cs), 1, 1);
  cfg.blockDim = dim3(kAttnThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cs;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LaunchScope ls(K_DECODE_ATTN, s);
  return cudaLaunchKernelEx(&cfg, decode_cluster_kernel<T, D, G, PAGED>, p, q, lengths, kn, vn, out, early);
}

template <typename T, int D, int G>
cudaError_t launch_typed(const DeviceProblem& p, const void* q, const int32_t* lengths, const void* k_new,
                         const void* v_new, void* out, cudaStream_t s, int early) {
  const unsigned char* kn = static_cast<const unsigned char*>(k_new);
  const unsigned char* vn = static_cast<const unsigned char*>(v_new);
  const int cs = cluster_size(p);
  if (cs > 0 && (cs <= 8 || (p.page_rows > 0 ? cluster16_fits<T, D, G, true>() : cluster16_fits<T, D, G, false>()))) {
    const T* qt = static_cast<const T*>(q);
    return p.page_rows > 0 ? launch_cluster<T, D, G, true>(p, cs, qt, lengths, kn, vn, static_cast<T*>(out), s, early)
                           : launch_cluster<T, D, G, false>(p, cs, qt, lengths, kn, vn, static_cast<T*>(out), s, early);
  }
  // persistent blocks: 16 per SM (measured best on B200 with 512-row items)
  int64_t grid = p.max_items < 16 * kSms ? p.max_items : 16 * kSms;
  if (grid < 1) grid = 1;
  cudaError_t e;
  {
    LaunchScope ls(K_DECODE_ATTN, s);
    const T* qt = static_cast<const T*>(q);
    e = p.page_rows > 0 ? launch_dependent(decode_attn_kernel<T, D, G, true>, (unsigned)grid, kAttnThreads, s, p, qt, lengths, kn,
                                           vn, static_cast<T*>(out), early)
                        : launch_dependent(decode_attn_kernel<T, D, G, false>, (unsigned)grid, kAttnThreads, s, p, qt, lengths, kn,
                                           vn, static_cast<T*>(out), early);
  }
  if (e != cudaSuccess) return e;
  {
    LaunchScope ls(K_DECODE_COMBINE, s);
    const int fused = k_new != nullptr ? 1 : 0;
    // units of at most 16 items each (32, if a block per head would be more than the GPU holds at once): a warp per head.
    // Otherwise a block per head; up to 16 of them per SM the variant that loads ahead (its blocks are resident within a
    // few waves)
    if (p.items_cap <= ((int64_t)p.view_U * G > 4 * kSms ? kDecodeFewItems : kDecodeFewItems / 2))
      e = launch_dependent(decode_combine_few_kernel<T, D, G>, (unsigned)((p.view_U * G + kCombineWarps - 1) / kCombineWarps),
                           kCombineThreads, s, p, lengths, fused, static_cast<T*>(out));
    else if (p.dec_tail != p.dec_shift)      // (fewer than 296 items after compression, so fewer units than that)
      e = launch_dependent(decode_combine_kernel<T, D, G, 8, true>, (unsigned)(p.view_U * G), kCombineThreads, s, p, lengths,
                           fused, static_cast<T*>(out));
    else if ((int64_t)p.view_U * G <= 16 * kSms)
      e = launch_dependent(decode_combine_kernel<T, D, G, 8, false>, (unsigned)(p.view_U * G), kCombineThreads, s, p, lengths,
                           fused, static_cast<T*>(out));
    else
      e = launch_dependent(decode_combine_kernel<T, D, G, 0, false>, (unsigned)(p.view_U * G), kCombineThreads, s, p, lengths,
                           fused, static_cast<T*>(out));
  }
  return e;
}

template <typename T, int D>
cudaError_t launch_group(const DeviceProblem& p, const void* q, const int32_t* lengths, const void* k_new,
                         const void* v_new, void* out, cudaStream_t s, int early) {
  switch (p.G) {
    case 1: return launch_typed<T, D, 1>(p, q, lengths, k_new, v_new, out, s, early);
    case 2: return launch_typed<T, D, 2>(p, q, lengths, k_new, v_new, out, s, early);
    case 4: return launch_typed<T, D, 4>(p, q, lengths, k_new, v_new, out, s, early);
    case 8: return launch_typed<T, D, 8>(p, q, lengths, k_new, v_new, out, s, early);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_decode(const DeviceProblem& p, int dtype, const void* q, const int32_t* lengths,
                          const void* k_new, const void* v_new, void* out, cudaStream_t s, bool early_unit_data) {
  // Reading lengths and page tables before the dependency wait is sound only if the kernel before this one in the
  // stream does not write them for these units; a caller's array of lengths is never read early.
  const int early = (early_unit_data && lengths == nullptr) ? 1 : 0;
  if (dtype == TASKKV_F32)
    return p.d == 64 ? launch_group<float, 64>(p, q, lengths, k_new, v_new, out, s, early)
                     : launch_group<float, 128>(p, q, lengths, k_new, v_new, out, s, early);
  return p.d == 64 ? launch_group<__nv_bfloat16, 64>(p, q, lengths, k_new, v_new, out, s, early)
                   : launch_group<__nv_bfloat16, 128>(p, q, lengths, k_new, v_new, out, s, early);
}

}  // namespace taskkv

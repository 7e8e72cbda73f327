// Selected-query bidirectional attention on the 5th-generation tensor cores (head_dim 128).
//
//   attn_fwd_tc    O = softmax(Q K^T / sqrt(Dh)) V and the log-sum-exp per (row, head).  One CTA per
//                  one or two tiles of up to 128 (selected row, query head) pairs of a K/V head and a
//                  sequence; keys stream in tiles of 128 through TMA.
//                  S = Q K^T is a tcgen05.mma into TMEM; softmax warps (one row per thread) read it
//                  with tcgen05.ld, write the bf16 probabilities back over the same TMEM columns and the
//                  PV product takes them from there as its A operand (V is the MN-major B operand straight
//                  from the TMA tile) and accumulates O in TMEM.
//   attn_abar_tc   Abar[r][j] = 1/Hq sum_h exp(s_h[r][j] - lse_h[r]) (Section 4.2): one pair of CTAs per
//                  (256 keys x up to 256 rows) loops over heads, S^T by tcgen05.mma, the sum over heads in
//                  registers in a fixed order (deterministic).
//
// Warp roles in both: warp 0 TMA producer, warp 1 MMA issuer + TMEM owner, warps 4..11 softmax/epilogue.
// No multicast load.  Every mbarrier wait is bounded (see gemm_tc.cu for the protocol).
#include <type_traits>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tc2_work.cuh"

namespace d2c {
namespace {

constexpr int AQ = 128, AKEYS = 128, ADH = 128;
constexpr int HALF_BYTES = 128 * 64 * 2;          // one 128-row x 64-column swizzled box: 16 KB
constexpr int TILE_BYTES = 2 * HALF_BYTES;        // 128 x 128 bf16
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

__device__ int g_attn_status[4];

// D (TMEM) (+)= A (TMEM) x B (shared memory): the probabilities stay in TMEM
__device__ __forceinline__ void umma_ts_e(uint32_t elected, uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                 "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// MN-major bf16 operand: 64 contiguous N elements per 128-byte row, 8 K-rows per 1024-byte group
// (stride offset), the next 64 N elements 16 KB further (leading offset).
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(HALF_BYTES >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// bf16 x bf16 -> fp32, M = 128, N = 128; bit 16 set: B is MN-major.
constexpr uint32_t kIdescKK = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescKMn = kIdescKK | (1u << 16);

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

struct AttnTcParams { AttnArgs a; int* status; int sm_count; int splits, head_groups, row_tile, pairs; int group, heads, kv_share, rows, split_last, places; };      // group: query heads of a tile, of the same K/V head; heads: such groups; kv_share: those of a K/V head; rows: selected rows of a query tile; places: tiles of a sequence's head that the grid has places for (0: numbered in turn)

// ------------------------------------------------------------------------------------------------
// Forward kernel.  One CTA owns up to two query tiles of one (sequence, K/V head), which share every K/V
// tile brought in by TMA.  A tile's 128 rows are `rows` selected rows x `group` query heads of that K/V head, the
// head the faster (18 x 7, two rows unused), or 128 selected rows of one head.  Each query tile has its own softmax warp
// group (4 warps, one row per thread) and its own TMEM columns: 128 for the scores S (overwritten in
// place by the bf16 probabilities P) and 128 for the output accumulator O, which stays in TMEM across
// the key tiles.  The running maximum is only raised when it grows by more than 2^8 (P stays exactly
// representable in bf16's exponent range); the rare raise rescales O in TMEM between two PV products.
constexpr int FWD_THREADS = 384;                  // warps 0..3: loader, MMA issuer, two idle; warps 4..11: softmax
constexpr float kRescaleStep = 8.f;
constexpr int kMaxSplits = 4;
// Of a tile's 128 keys, those whose probabilities are handed over first.  The products of the others and the next scores are what a
// query tile waits for: 3240 clocks a pair of score tiles with 64 first, of which the special function unit takes 2048 and the tensor
// cores as many.  Forward alone, us, with 32 / 64 / 96 first: 976 rows of four sequences x 1536 keys x 28 heads 105.4 / 103.8 / 100.2,
// 797 x 797 x 32 20.5 / 20.3 / 19.6, 147 of four x 1187 x 28 28.3 / 28.2 / 27.3, 300 of five x 3071 x 32 143.4 / 141.9 / 138.3; one
// query tile a CTA (489 x 768 x 32) 13.0 / 12.8 / 12.8.
constexpr int kFirstKeys = 96;

// Packed pairs of fp32 for Blackwell's two-wide FMA-pipe instructions: one issue slot for two elements.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
               "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                 "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
                 "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
                 "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory");
}

// Items are numbered sequence by sequence, `mine` of them for this lane's sequence (lane l: sequence b0 + l): the lane whose items include
// the i-th, which becomes its number among those, or -1 and i less all of them.  A warp finds it together.
__device__ __forceinline__ int lane_of_item(int mine, int& i) {
  int sum = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, sum, o);
    if ((int)(threadIdx.x & 31) >= o) sum += up;
  }
  const unsigned behind = __ballot_sync(0xffffffffu, i < sum);
  const int at = behind ? __ffs(behind) - 1 : 31;
  i -= __shfl_sync(0xffffffffu, behind ? sum - mine : sum, at);
  return behind ? at : -1;
}

// What a CTA of the forward works on: sequence, K/V head, first row, rows (0: nothing).  By a whole warp.  A call, as its registers would
// otherwise be taken from the softmax warps', which then spill.
// The grid has room for all rows of all sequences, and a CTA without any still holds an SM, of whose shared memory it wants nearly all,
// for a microsecond.  So the live ones are numbered in turn and the others come behind them; by their places in a grid of (tiles, heads,
// sequences), where they stood between, us: 147 rows of four sequences x 1187 keys x 28 heads 33.1 -> 24.6, 260 of eight x 700 54.0 ->
// 49.0, 300 of five x 3071 x 32 144.4 -> 133.0, 2880 of two x 4096 348.5 -> 345.5, 976 of four x 1536 and 797 x 797 no difference.  (Items
// of two tiles first, those of one behind them: 142 where it is 134, as a head's keys then come out of the L2 no longer.)
template <bool kGroup, bool kSplitLast>
__device__ __noinline__ int4 forward_item(const int32_t* row_off, int batch, int heads, int rows_, int sm_count) {
  const int rows = kGroup ? rows_ : AQ;
  const int lane = threadIdx.x & 31;
  int i = blockIdx.x, all = 0, pairs = 0, half = -1;                // tiles, and pairs of them
  const auto tiles_of = [&](int n) { return kGroup ? div24(n + rows - 1, rows) : (n + AQ - 1) / AQ; };
  // What is left over behind whole waves of pairs, where it is so little that its tiles can have an SM each, is split into tiles: a pair
  // takes 1.6 times as long as a tile.  Forward alone, us: 976 rows of four sequences x 1536 keys x 28 heads over 4 (448 pairs) 93.6 -> 88.0,
  // 420 of three x 1100 x 32 42.5 -> 39.3, 300 of five x 3071 133.0 -> 129.9.
  const auto split_last = [&]() {
    const int whole = div24(pairs, sm_count) * sm_count;
    if (all > sm_count && 2 * (pairs - whole) <= sm_count && i >= whole) { half = (i - whole) & 1; i = whole + ((i - whole) >> 1); }
  };
  const auto item_of = [&](int b, int g, int first, int n, int r, int width) {
    if (kSplitLast && half >= 0) { r += half * rows; width = 1; }
    return make_int4(b, g, first + r, min(width * rows, n - r));
  };
  if (batch == 1) {                                                 // (without the scan: 0.3 us of a launch)
    const int first = row_off[0], n = row_off[1] - first, tiles = tiles_of(n), width = tiles * heads > sm_count ? 2 : 1;
    all = tiles * heads; pairs = ((tiles + 1) >> 1) * heads;
    if (kSplitLast) split_last();
    const int of = max((tiles + width - 1) >> (width - 1), 1), g = div24(i, of);
    return g < heads ? item_of(0, g, first, n, (i - g * of) * width * rows, width) : make_int4(0, 0, 0, 0);
  }
  int first = 0, n = 0, tiles = 0;
  const auto load = [&](int b0) {
    first = b0 + lane < batch ? row_off[b0 + lane] : 0; n = b0 + lane < batch ? row_off[b0 + lane + 1] - first : 0; tiles = tiles_of(n);
  };
  const int last = (batch - 1) & ~31;                               // (up to 32 sequences are loaded once)
  for (int b0 = 0; b0 <= last; b0 += 32) {
    load(b0);
    all += __reduce_add_sync(0xffffffffu, tiles * heads);
    if (kSplitLast) pairs += __reduce_add_sync(0xffffffffu, ((tiles + 1) >> 1) * heads);
  }
  const int width = all > sm_count ? 2 : 1;                         // tiles of an item
  if (kSplitLast) split_last();
  for (int b0 = 0; b0 <= last; b0 += 32) {
    if (last > 0) load(b0);
    const int per = (tiles + width - 1) >> (width - 1), at = lane_of_item(per * heads, i);      // per: items of a head
    if (at < 0) continue;
    const int of = __shfl_sync(0xffffffffu, per, at), g = div24(i, of);
    return item_of(b0 + at, g, __shfl_sync(0xffffffffu, first, at), __shfl_sync(0xffffffffu, n, at), (i - g * of) * width * rows, width);
  }
  return make_int4(0, 0, 0, 0);
}

// kGroup: a tile has several query heads (one: the tile's divisions by their number fold away, 0.3 us of a CTA).
// kOne: there are places for all tiles, so that a CTA has one tile at most, at its place.  (With the schedule for two in it as well a launch takes
// 0.3 to 0.9 us longer: it is larger, and runs once.  Two layers of d 512, 194 rows of 570 positions 113.9 / 112.5 us a step, all of 300 in
// eight sequences 178.7 / 176.7, four of d 4096, 40 rows of eight x 142 616 / 611.)
template <bool kSplit, bool kGroup, bool kOne>
__global__ void __launch_bounds__(FWD_THREADS, 1)
attn_fwd_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
            const __grid_constant__ CUtensorMap tmV, const AttnTcParams p) {
  pdl_prologue();
  const AttnArgs& a = p.a;
  const int group = kGroup ? p.group : 1, tile_rows = kGroup ? p.rows : AQ;
  // With few selected rows every 128-row tile gets a CTA of its own (more SMs busy); otherwise a CTA
  // takes two tiles, which halves the K/V traffic per row and keeps both softmax warp groups busy.
  // With so few that SMs would idle all the same, the CTAs of a cluster share one tile's keys (p.splits of them).
  const int splits = kSplit ? p.splits : 1, part = kSplit ? (int)blockIdx.x : 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // What this CTA works on: sequence, K/V head, first row, rows (none: nothing).  One warp works it out, and the softmax warps read it where
  // they need it: held from here on it made them spill.
  __shared__ int s_item[4];
  volatile int* item = s_item;
  if constexpr (kSplit) {
    // The row tile is the slowest index, so that the live ones start first.  Without kOne the grid has room for half of the tiles only that
    // there can be: with more rows than that every CTA takes two.  (Its other CTAs find nothing to do.)
    const int b = (int)blockIdx.z % a.batch, r0 = a.row_off[b], nb = a.row_off[b + 1] - r0;
    const int width = !kOne && nb > p.places * tile_rows ? 2 * tile_rows : tile_rows, at = (int)blockIdx.z / a.batch * width;
    if (at >= nb) return;                                           // uniform in the cluster: nothing allocated yet
    if (threadIdx.x == 0) { item[0] = b; item[1] = blockIdx.y; item[2] = r0 + at; item[3] = min(width, nb - at); }
  } else if constexpr (kOne) {
    // (by its place among `places` of each head: the numbering takes a CTA of several sequences 0.5 us)
    const int bg = div24(blockIdx.x, p.places), b = div24(bg, p.heads), r0 = a.row_off[b], at = ((int)blockIdx.x - bg * p.places) * tile_rows;
    const int nrows = min(tile_rows, a.row_off[b + 1] - r0 - at);
    if (nrows <= 0) return;
    if (threadIdx.x == 0) { item[0] = b; item[1] = bg - b * p.heads; item[2] = r0 + at; item[3] = nrows; }
  } else if (warp == 0) {
    const int4 it = p.split_last ? forward_item<kGroup, true>(a.row_off, a.batch, p.heads, tile_rows, p.sm_count)
                                 : forward_item<kGroup, false>(a.row_off, a.batch, p.heads, tile_rows, p.sm_count);
    if (lane == 0) { item[0] = it.x; item[1] = it.y; item[2] = it.z; item[3] = it.w; }
  }
  const int L = a.seq_len, tiles = (L + AKEYS - 1) / AKEYS;
  const int first = kSplit ? tiles * part / splits : 0, T = kSplit ? tiles * (part + 1) / splits - first : tiles;      // this CTA's key tiles (at least one)
  int* const status = p.status;                                     // (from the arguments at each use: held, it is two registers too many)

  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = ((uint32_t)__cvta_generic_to_shared(smem_raw) + 1023u) & ~1023u;
  auto sQ = [&](int q) { return sbase + q * TILE_BYTES; };
  auto sK = [&](int s) { return sbase + (2 + 2 * s) * TILE_BYTES; };
  auto sV = [&](int s) { return sbase + (3 + 2 * s) * TILE_BYTES; };
  // barriers: 0 q_full | 1,2 k_full | 3,4 v_full | 5,6 kv_empty | 7,8 s_full[q] | 9,10 p_full[q], the first keys | 11,12 o_full[q] |
  // 13,14 p_full[q], the others
  __shared__ __align__(8) uint64_t bars[15];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(bars);
  auto B = [&](int i) { return bar0 + 8u * i; };
  if (threadIdx.x == 64) {
    for (int i = 0; i < 9; ++i) mbar_init(B(i), 1);
    mbar_init(B(9), 4); mbar_init(B(10), 4);
    mbar_init(B(11), 1); mbar_init(B(12), 1);
    mbar_init(B(13), 4); mbar_init(B(14), 4);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) { tmem_alloc((uint32_t)__cvta_generic_to_shared(&tmem_slot), 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (!kSplit && !kOne && item[3] <= 0) {
    if (warp == 1) tmem_dealloc(tmem_slot, 512);
    return;
  }
  const int nq = !kOne && item[3] > tile_rows ? 2 : 1;                          // live query tiles
  const uint32_t tm = tmem_slot;                                    // tile q: S/P at q*256, O at q*256 + 128
  volatile int* abortp = &abort_flag;

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
  if (warp == 0) {
    if (lane == 0) {
      const int h = item[1], g = kGroup || p.kv_share == 1 ? h : h / p.kv_share, r0 = item[2], kv_row0 = item[0] * a.cache_seq + first * AKEYS;
      mbar_expect_tx(B(0), nq * tile_rows * group * ADH * 2);
      for (int q = 0; q < nq; ++q) {
        if constexpr (kGroup) {
          tma_load_3d(sQ(q), &tmQ, 0, h * group, r0 + q * tile_rows, B(0));
          tma_load_3d(sQ(q) + HALF_BYTES, &tmQ, 64, h * group, r0 + q * tile_rows, B(0));
        } else {
          tma_load_2d(sQ(q), &tmQ, h * ADH, r0 + q * AQ, B(0));
          tma_load_2d(sQ(q) + HALF_BYTES, &tmQ, h * ADH + 64, r0 + q * AQ, B(0));
        }
      }
      int issued = 0;
      for (int j = 0; j < T; ++j) {
        const int s = j & 1, u = j >> 1;
        if (!mbar_wait(B(5 + s), (u & 1) ^ 1, abortp, status, 11)) break;
        mbar_expect_tx(B(1 + s), TILE_BYTES);
        tma_load_2d(sK(s), &tmK, g * ADH, kv_row0 + j * AKEYS, B(1 + s));
        tma_load_2d(sK(s) + HALF_BYTES, &tmK, g * ADH + 64, kv_row0 + j * AKEYS, B(1 + s));
        mbar_expect_tx(B(3 + s), TILE_BYTES);
        tma_load_2d(sV(s), &tmV, g * ADH, kv_row0 + j * AKEYS, B(3 + s));
        tma_load_2d(sV(s) + HALF_BYTES, &tmV, g * ADH + 64, kv_row0 + j * AKEYS, B(3 + s));
        issued = j + 1;
      }
      if (*abortp) {
        const long long t0 = clock64();
        while (!mbar_try_wait(B(0), 0) && clock64() - t0 < kWaitCycles) {}
        for (int j = max(0, issued - 2); j < issued; ++j) {
          const long long t1 = clock64();
          while (!(mbar_try_wait(B(1 + (j & 1)), (j >> 1) & 1) && mbar_try_wait(B(3 + (j & 1)), (j >> 1) & 1)) &&
                 clock64() - t1 < kWaitCycles) {}
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      const uint32_t el = elect_one();
      auto issue_s = [&](int q, int j) {                            // S_{q,j} = Q_q K_j^T
        const int s = j & 1;
#pragma unroll
        for (int i = 0; i < ADH / 16; ++i) {
          const uint32_t off = (i >> 2) * HALF_BYTES;
          umma_ss_e(el, tm + q * 256, smem_desc_sw128(sQ(q) + off) + 2 * (i & 3), smem_desc_sw128(sK(s) + off) + 2 * (i & 3), kIdescKK, i != 0);
        }
        umma_commit_e(el, B(7 + q));
      };
      bool ok = mbar_wait_warp(B(0), 0, abortp, status, 12) && mbar_wait_warp(B(1), 0, abortp, status, 13);
      if (nq == 1) {
        // One live query tile: the second tile's TMEM columns are free, so the scores of key tile j + 1 are
        // computed there while the softmax warps work on tile j (S/P buffer = j & 1, O stays in the first half).
        auto issue_s1 = [&](int j) {
          const int s = j & 1;
#pragma unroll
          for (int i = 0; i < ADH / 16; ++i) {
            const uint32_t off = (i >> 2) * HALF_BYTES;
            umma_ss_e(el, tm + s * 256, smem_desc_sw128(sQ(0) + off) + 2 * (i & 3), smem_desc_sw128(sK(s) + off) + 2 * (i & 3), kIdescKK, i != 0);
          }
          umma_commit_e(el, B(7 + s));
        };
        if (ok) {
          tc_fence_after();
          issue_s1(0);
        }
        for (int j = 0; j < T && ok; ++j) {
          const int s = j & 1, u = j >> 1;
          if (j + 1 < T) {
            if (!mbar_wait_warp(B(1 + ((j + 1) & 1)), ((j + 1) >> 1) & 1, abortp, status, 16)) { ok = false; break; }
            tc_fence_after();
            issue_s1(j + 1);                                        // its buffer held P_{j-1}, consumed by the product issued before
          }
          if (!mbar_wait_warp(B(9 + s), u & 1, abortp, status, 14)) { ok = false; break; }
          if (!mbar_wait_warp(B(3 + s), u & 1, abortp, status, 15)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int i = 0; i < kFirstKeys / 16; ++i)
            umma_ts_e(el, tm + 128, tm + s * 256 + 8 * i, desc_mnmajor(sV(s) + i * 2048), kIdescKMn, (j | i) != 0);
          if (!mbar_wait_warp(B(13 + s), u & 1, abortp, status, 14)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int i = kFirstKeys / 16; i < AKEYS / 16; ++i)
            umma_ts_e(el, tm + 128, tm + s * 256 + 8 * i, desc_mnmajor(sV(s) + i * 2048), kIdescKMn, 1);
          umma_commit_e(el, B(11));
          umma_commit_e(el, B(5 + s));
        }
        ok = false;                                                 // done: skip the two-tile schedule below
      } else if (ok) {
        tc_fence_after();
        for (int q = 0; q < nq; ++q) issue_s(q, 0);
      }
      for (int j = 0; j < T && ok; ++j) {
        const int s = j & 1, u = j >> 1;
        for (int q = 0; q < nq && ok; ++q) {
          if (!mbar_wait_warp(B(9 + q), j & 1, abortp, status, 14)) { ok = false; break; }
          if (q == 0 && !mbar_wait_warp(B(3 + s), u & 1, abortp, status, 15)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int i = 0; i < kFirstKeys / 16; ++i)                     // O_q += P_{q,j} (TMEM, 8 columns per 16 keys) x V_j
            umma_ts_e(el, tm + q * 256 + 128, tm + q * 256 + 8 * i, desc_mnmajor(sV(s) + i * 2048), kIdescKMn, (j | i) != 0);
          if (q == 0 && j + 1 < T && !mbar_wait_warp(B(1 + ((j + 1) & 1)), ((j + 1) >> 1) & 1, abortp, status, 16)) { ok = false; break; }
          if (!mbar_wait_warp(B(13 + q), j & 1, abortp, status, 14)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int i = kFirstKeys / 16; i < AKEYS / 16; ++i)
            umma_ts_e(el, tm + q * 256 + 128, tm + q * 256 + 8 * i, desc_mnmajor(sV(s) + i * 2048), kIdescKMn, 1);
          umma_commit_e(el, B(11 + q));
          if (q == nq - 1) umma_commit_e(el, B(5 + s));                   // both products of tile j issued: K/V stage free when done
          if (j + 1 < T) {
            issue_s(q, j + 1);                                      // after PV_{q,j} in program order: P_{q,j} is consumed first
          }
        }
      }
    }
    __syncwarp();
  } else if (warp >= 4) {
    // 232 registers for the softmax threads, taken from the other four warps' (384 x 168 at launch = 128 x 40 + 256 x 232)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    const int q = (warp - 4) >> 2;                                  // softmax warp group = query tile
    if (q < nq) {
      const int quarter = warp & 3, lrow = q * AQ + quarter * 32 + lane;
      const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
      const bool dbuf = kOne || item[3] <= tile_rows;                            // one query tile: S/P alternate between the TMEM halves
      const uint32_t to = tm + q * 256 + 128 + lane_base;
      const float sc = kLog2e * rsqrtf((float)ADH);
      float m_used = -INFINITY, l = 0.f;
      bool ok = true;
      for (int j = 0; j < T && ok; ++j) {
        const int sp = dbuf ? (j & 1) : q;                          // S/P buffer of this tile
        const uint32_t ts = tm + sp * 256 + lane_base;
        // a wait that gave up ends the loop for the whole warp: the tcgen05.ld / st below are warp-collective
        if (!__all_sync(0xffffffffu, mbar_wait(B(7 + sp), (dbuf ? (j >> 1) : j) & 1, abortp, status, 18))) { ok = false; break; }
        tc_fence_after();
        const int key0 = (first + j) * AKEYS;
        const bool full = key0 + AKEYS <= L;
        uint32_t sv[4][32];                                         // the whole score row of this thread
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(ts + c * 32, sv[c]);
        tmem_ld_wait();
        if (!full) {                                                // last, ragged key tile: keys past L score -inf (probability 0)
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (key0 + c * 32 + i >= L) sv[c][i] = __float_as_uint(-INFINITY);
        }
        // Probabilities are taken relative to the maximum used so far, without waiting for this tile's own: the special
        // function unit (16 exponentials a clock, 1024 clocks a tile) then works while the maximum is found.  Only if
        // that has grown by more than 2^8 are the first keys done again, relative to the new one.
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        auto max32 = [&](int c) {                                   // three-input maximum: two scores per instruction
#pragma unroll
          for (int i = 0; i < 32; i += 2) mx4[(i >> 1) & 3] = fmax3(mx4[(i >> 1) & 3], __uint_as_float(sv[c][i]), __uint_as_float(sv[c][i + 1]));
        };
        auto row_max = [&]() { return fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * sc; };
        // scale-and-subtract and the row sums run two elements per instruction (fma / add .f32x2)
        unsigned long long rs2[4];                                  // packed pairs of partial row sums
        const unsigned long long sc2 = pack2(sc, sc);
        uint32_t pk[AKEYS / 32][16];
        // probabilities of the keys [16 b0, 16 b1), rounded to bf16, in batches of 16: a batch is summed and rounded behind the
        // next one's exponentials, so that nothing waits for a result of the special function unit
        auto some_keys = [&](auto b0_, auto b1_, bool with_max) {
          constexpr int b0 = decltype(b0_)::value, b1 = decltype(b1_)::value;
          const unsigned long long nm2 = pack2(-m_used, -m_used);
          float pp[2][16];
#pragma unroll
          for (int b = b0; b < b1 + 1; ++b) {
            if (b < b1) {
              float x[16];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const int c = b >> 1, e = (b & 1) * 16 + 2 * i;
                unpack2(fma2(pack2(__uint_as_float(sv[c][e]), __uint_as_float(sv[c][e + 1])), sc2, nm2), x[2 * i], x[2 * i + 1]);
              }
#pragma unroll
              for (int i = 0; i < 16; ++i) pp[b & 1][i] = exp2f(x[i]);
              if (with_max && b < 4) max32(b);
            }
            if (b > b0) {
              const int d = b - 1;
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                rs2[i & 3] = add2(rs2[i & 3], pack2(pp[d & 1][2 * i], pp[d & 1][2 * i + 1]));
                pk[d >> 1][(d & 1) * 8 + i] = pack_bf16(pp[d & 1][2 * i], pp[d & 1][2 * i + 1]);
              }
            }
          }
        };
        auto zero_sums = [&]() { rs2[0] = rs2[1] = rs2[2] = rs2[3] = 0ull; };      // (the bits of 0.f are 0)
        zero_sums();
        constexpr std::integral_constant<int, 0> kBegin{};
        constexpr std::integral_constant<int, kFirstKeys / 16> kMid{};
        constexpr std::integral_constant<int, AKEYS / 16> kEnd{};
        if (j > 0) some_keys(kBegin, kMid, true);
        else { max32(0); max32(1); max32(2); max32(3); }
        const float mx = row_max();
        const bool raise = mx > m_used + kRescaleStep;              // always true on the first tile
        if (__any_sync(0xffffffffu, raise)) {
          const float alpha = raise ? exp2f(m_used - mx) : 1.f;     // first tile: exp2(-inf) = 0
          if (raise) m_used = mx;
          l *= alpha;
          if (j > 0) {                                              // O holds the sum of tiles 0..j-1: rescale it in place
            if (!__all_sync(0xffffffffu, mbar_wait(B(11 + q), (j - 1) & 1, abortp, status, 17))) { ok = false; break; }
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t v[32];
              tmem_ld32(to + c * 32, v);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
              tmem_st32(to + c * 32, v);
            }
            tmem_st_wait();
          }
          zero_sums();
          some_keys(kBegin, kMid, false);
        }
        // written back as bf16 over the scores: the product with V starts on the first keys while the others' are worked out.  (Not
        // stored among the exponentials: the kernel then spills, 20 to 24 bytes by chance of what stands elsewhere in it, and is up to
        // 10 % slower: 976 rows of four sequences x 1536 keys 100 us, 101 or 112 that way.)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          if (hf == 1) some_keys(kMid, kEnd, false);
#pragma unroll
          for (int c = hf ? kFirstKeys / 32 : 0; c < (hf ? AKEYS : kFirstKeys) / 32; ++c) tmem_st16(ts + c * 16, pk[c]);
          tmem_st_wait();
          // Behind the loop the last product is waited for, and a parity wait only tells a phase from the one before it.  The
          // last scores do not wait for the product before the last (its V may come in late), so that one is waited for
          // here, where the last cannot be done yet: it needs these keys.
          if (hf == 1 && j > 0 && j == T - 1) ok = __all_sync(0xffffffffu, mbar_wait(B(11 + q), (j - 1) & 1, abortp, status, 17));
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(B((hf ? 13 : 9) + sp));
        }
        float rs4[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) { float lo, hi; unpack2(rs2[t], lo, hi); rs4[t] = lo + hi; }
        l += (rs4[0] + rs4[1]) + (rs4[2] + rs4[3]);
      }
      // (A warp without live rows goes all the way with the others: one that skipped the wait above passed this one a phase early, and
      // was no faster: 976 rows of four sequences x 1536 keys 101.2 -> 100.4 us, 300 of five x 3071 139.9 -> 139.1, 147 of four x 1187
      // 27.0 -> 27.3.)
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(B(11 + q), (T - 1) & 1, abortp, status, 19));
      tc_fence_after();
      if (kSplit && ok) {
        // this CTA's share of the sum and what it is relative to, for the meeting below: over the Q tiles and the first K/V stage, a
        // row's 16-byte pieces swizzled over the banks (every MMA of this query tile has read its operands; see the wait)
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t v[32];
          tmem_ld32(to + c * 32, v);
          tmem_ld_wait();
#pragma unroll
          for (int t = 0; t < 8; ++t)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sbase + (uint32_t)(lrow * 512 + (((c * 8 + t) ^ (lrow & 31)) << 4))),
                         "r"(v[4 * t]), "r"(v[4 * t + 1]), "r"(v[4 * t + 2]), "r"(v[4 * t + 3]) : "memory");
        }
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(sK(1) + (uint32_t)lrow * 8u), "f"(m_used), "f"(l) : "memory");
      } else if (ok) {
        // Through this warp's part of its Q tile, which every MMA has read: a row's 16-byte pieces, swizzled, go in by rows and
        // come out as whole rows.  (Each thread storing its own row, 16 bytes at a time: 976 rows of four sequences x 1536 keys 107.5 us,
        // 100.7 this way, 797 x 797 20.4 and 19.9, 147 of four x 1187 28.0 and 27.5.)
        // A tile's row is (selected row, head of the group), the head the faster: its outputs lie one behind the other too.
        const int live = min(item[3] - q * tile_rows, tile_rows) * group, m0 = quarter * 32;
        const size_t first_out = (size_t)(item[2] + q * tile_rows) * a.hq + item[1] * group;
        const float inv = 1.f / l;
        const uint32_t stage = sQ(q) + (uint32_t)(quarter * 32) * 256u;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint32_t v[32];
          tmem_ld32(to + c * 32, v);
          tmem_ld_wait();
#pragma unroll
          for (int t = 0; t < 4; ++t)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stage + (uint32_t)(lane * 256 + (((c * 4 + t) ^ (lane & 15)) << 4))),
                         "r"(pack_bf16(__uint_as_float(v[8 * t + 0]) * inv, __uint_as_float(v[8 * t + 1]) * inv)),
                         "r"(pack_bf16(__uint_as_float(v[8 * t + 2]) * inv, __uint_as_float(v[8 * t + 3]) * inv)),
                         "r"(pack_bf16(__uint_as_float(v[8 * t + 4]) * inv, __uint_as_float(v[8 * t + 5]) * inv)),
                         "r"(pack_bf16(__uint_as_float(v[8 * t + 6]) * inv, __uint_as_float(v[8 * t + 7]) * inv)) : "memory");
        }
        __syncwarp();
        int sel = kGroup ? div24(m0 + (lane >> 4), group) : m0 + (lane >> 4), head = m0 + (lane >> 4) - sel * group;
        const int step = 2 / min(group, 4), rest = group > 2 ? 2 : 0;      // two of the tile's rows on, in selected rows and heads
#pragma unroll 4
        for (int i = 0; i < 16; ++i) {
          const int r = 2 * i + (lane >> 4), pc = lane & 15;
          uint4 w;
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                       : "r"(stage + (uint32_t)(r * 256 + ((pc ^ (r & 15)) << 4))) : "memory");
          if (m0 + r < live) reinterpret_cast<uint4*>(a.o + (first_out + (size_t)sel * a.hq + head) * ADH)[pc] = w;
          sel += step; head += rest;
          if (kGroup && head >= group) { head -= group; ++sel; }
        }
        sel = kGroup ? div24(m0 + lane, group) : m0 + lane;
        if (m0 + lane < live) a.lse[first_out + (size_t)sel * a.hq + (m0 + lane - sel * group)] = (m_used + log2f(l)) * kLn2;
      }
    }
  }
  if (kSplit) {
    __syncwarp();
    cluster_sync_all();
    if (warp >= 4 && !*abortp) {
      // this CTA's share of the tile's rows, a warp a row: the parts' sums relative to the largest of their maxima
      const int first_live = min(item[3], tile_rows) * group, live = first_live + (!kOne && item[3] > tile_rows ? (item[3] - tile_rows) * group : 0);
      const int ra = live * part / splits, rb = live * (part + 1) / splits;
      for (int n = ra + (warp - 4); n < rb; n += 8) {
        const int q = !kOne && n >= first_live ? 1 : 0, mine = n - q * first_live, r = q * AQ + mine, sel = kGroup ? div24(mine, group) : mine;
        const size_t at = (size_t)(item[2] + q * tile_rows + sel) * a.hq + item[1] * group + mine - sel * group;
        float pm[kMaxSplits], pl[kMaxSplits], m = -INFINITY, l = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), x[kMaxSplits];
        const uint32_t o_at = sbase + (uint32_t)(r * 512 + ((lane ^ (r & 31)) << 4)), m_at = sK(1) + (uint32_t)r * 8u;
#pragma unroll
        for (int s = 0; s < kMaxSplits; ++s) {
          pm[s] = -INFINITY; pl[s] = 0.f; x[s] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (s < splits) {
            uint32_t ro, rm;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ro) : "r"(o_at), "r"((uint32_t)s));
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rm) : "r"(m_at), "r"((uint32_t)s));
            asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(pm[s]), "=f"(pl[s]) : "r"(rm) : "memory");
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[s].x), "=f"(x[s].y), "=f"(x[s].z), "=f"(x[s].w) : "r"(ro) : "memory");
          }
        }
#pragma unroll
        for (int s = 0; s < kMaxSplits; ++s) m = fmaxf(m, pm[s]);
#pragma unroll
        for (int s = 0; s < kMaxSplits; ++s) {                      // in part order (deterministic)
          const float w = exp2f(pm[s] - m);
          l = fmaf(pl[s], w, l);
          acc.x = fmaf(x[s].x, w, acc.x); acc.y = fmaf(x[s].y, w, acc.y); acc.z = fmaf(x[s].z, w, acc.z); acc.w = fmaf(x[s].w, w, acc.w);
        }
        const float inv = 1.f / l;
        reinterpret_cast<uint2*>(a.o + at * ADH)[lane] = make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        if (lane == 0) a.lse[at] = (m + log2f(l)) * kLn2;
      }
    }
    __syncwarp();
    cluster_sync_all();                                             // nobody leaves while its part may still be read
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tm, 512); }
}

// ------------------------------------------------------------------------------------------------
// Head-averaged probabilities.  The keys are the M operand and the selected rows the N operand: a pair of CTAs (two SMs,
// cta_group::2) owns 256 keys, 128 in each CTA's TMEM lanes, and a tile of up to 256 rows, any multiple of 16, of whose Q
// each CTA brings in half.  Per head S^T = K Q^T goes to TMEM (two buffers) and the epilogue adds exp(s - lse) to sums
// in registers, in head order (deterministic).
// The kernel is bound by the special function unit (1024 clocks per 128 x 128 scores) as long as the operands come in
// fast enough: 64 KB a head and CTA for two such tiles.  One CTA with its own 128 x 128 tile needs 64 KB for one, which at
// the 9.6 TB/s the L2 delivers was the limit.  And this way round only the keys are padded: rows come in sixteens.
// Where the tiles are too few for the GPU the heads are shared by two or four pairs of one cluster; their sums meet in
// shared memory and each CTA adds (in head order) and writes its share of the rows.
constexpr int ABS = 3;                             // stages of the Q ring and of the K ring
constexpr int ABAR_THREADS = 384;                  // warps 0..3: loader, MMA issuer, two idle; warps 4..11: epilogue
constexpr int N_QBOX = 6;                          // heights of the Q boxes (rows per CTA)
__host__ __device__ constexpr int q_box_rows(int i) { return i == 0 ? 16 : i == 1 ? 32 : i == 2 ? 48 : i == 3 ? 64 : i == 4 ? 96 : 128; }
constexpr int ABAR_MAX_ROWS = 256;                 // rows of a tile; the staged log-sum-exp holds that many for 32 heads
constexpr int kAbarSmem = 2 * ABS * TILE_BYTES + 1024 + ABAR_MAX_ROWS * 32 * 4 + 128;   // (a block of 32 rows may read past the last tile's end)

struct AbarMaps { CUtensorMap k, q[N_QBOX]; };
struct Item { int b, key0, w, r0, nrows, bi; };      // sequence, this CTA's first key, width and rows of the tile, height of the Q box

// A tile of sequence t.b's rows (the sequence's rows in tiles of almost equal width) and 256 keys; false if there is no such tile.
__device__ __forceinline__ bool cut_item(const AttnTcParams& p, int first, int nb, int tile, int keys, uint32_t rank, Item& t) {
  const int units = (nb + 15) >> 4;
  const int tiles = div24(units * 16 + p.row_tile - 1, p.row_tile);
  if (tile >= tiles) return false;
  const int ub = div24(units, tiles), ur = units - ub * tiles, col0 = 16 * (tile * ub + min(tile, ur));
  t.w = 16 * (ub + (tile < ur ? 1 : 0));
  t.r0 = first + col0; t.nrows = min(t.w, nb - col0);
  t.key0 = (keys * 2 + (int)rank) * AKEYS;
  t.bi = 0;
  while (t.bi + 1 < N_QBOX && q_box_rows(t.bi) < (t.w >> 1)) ++t.bi;
  return true;
}
__device__ __forceinline__ int items_of(const AttnTcParams& p, int nb) {
  return (p.a.seq_len + 2 * AKEYS - 1) / (2 * AKEYS) * div24(((nb + 15) & ~15) + p.row_tile - 1, p.row_tile);
}
// The cluster's item where the live ones are numbered in turn, so that no cluster without one stands between them.  By whole warps.
__device__ __forceinline__ bool first_item(const AttnTcParams& p, int cluster, uint32_t rank, Item& t) {
  const int kpairs = (p.a.seq_len + 2 * AKEYS - 1) / (2 * AKEYS);
  int i = cluster;
  for (int b0 = 0; b0 < p.a.batch; b0 += 32) {
    const int b = b0 + (threadIdx.x & 31), first = b < p.a.batch ? p.a.row_off[b] : 0, nb = b < p.a.batch ? p.a.row_off[b + 1] - first : 0;
    const int at = lane_of_item(items_of(p, nb), i);
    t.b = b0 + at;
    const int tile = div24(max(i, 0), kpairs);
    if (at >= 0) return cut_item(p, __shfl_sync(0xffffffffu, first, at), __shfl_sync(0xffffffffu, nb, at), tile, i - tile * kpairs, rank, t);
  }
  return false;
}
// With `pairs` clusters that stay, each takes every pairs-th item: its n-th.
__device__ __forceinline__ bool nth_item(const AttnTcParams& p, int n, uint32_t rank, Item& t) {
  const int kpairs = (p.a.seq_len + 2 * AKEYS - 1) / (2 * AKEYS);
  int i = (int)(blockIdx.x >> 1) + n * p.pairs;
  for (t.b = 0; t.b < p.a.batch; ++t.b) {
    const int first = p.a.row_off[t.b], nb = p.a.row_off[t.b + 1] - first, of = items_of(p, nb);
    if (i < of) return cut_item(p, first, nb, i / kpairs, i % kpairs, rank, t);
    i -= of;
  }
  return false;
}

// How the clusters come to their items: each its own by its place in the grid, or numbered in turn, or a.pairs clusters do all of them.
enum AbarForm { ABAR_GRID = 0, ABAR_IN_TURN = 1, ABAR_STAY = 2 };
template <AbarForm kForm>
__global__ void __launch_bounds__(ABAR_THREADS, 1)
attn_abar_tc(const __grid_constant__ AbarMaps maps, const AttnTcParams p) {
  constexpr bool kStay = kForm == ABAR_STAY;
  pdl_prologue();
  const AttnArgs& a = p.a;
  const int L = a.seq_len;
  const int hgs = kStay ? 1 : p.head_groups;                        // pairs of this cluster, each with its own heads
  const uint32_t crank = cluster_ctarank(), rank = crank & 1;       // rank: inside the pair
  const int hg = (int)crank >> 1;
  const uint16_t both = (uint16_t)(3u << (crank & ~1u));            // the pair, for multicast commits
  const int nh = a.hq / hgs, h_first = hg * nh;                     // this pair's heads (whole kv groups)
  Item it;
  // (return: the whole cluster)
  if constexpr (kForm == ABAR_STAY) {
    if (!nth_item(p, 0, rank, it)) return;
  } else if constexpr (kForm == ABAR_IN_TURN) {
    if (!first_item(p, (int)blockIdx.x >> (hgs == 4 ? 3 : hgs), rank, it)) return;
  } else {
    it.b = blockIdx.z;
    const int first = a.row_off[it.b];
    if (!cut_item(p, first, a.row_off[it.b + 1] - first, blockIdx.y, (int)blockIdx.x / (2 * hgs), rank, it)) return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = a.hq / a.hkv;
  int* const status = p.status;

  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = ((uint32_t)__cvta_generic_to_shared(smem_raw) + 1023u) & ~1023u;
  auto sK = [&](int s) { return base + s * TILE_BYTES; };           // ABS key stages, then ABS query stages, then -lse * log2(e)
  auto sQ = [&](int s) { return base + (ABS + s) * TILE_BYTES; };
  const uint32_t s_lse = base + 2 * ABS * TILE_BYTES;               // [head][w]
  // barriers: q_full[ABS] | k_full[ABS] | q_empty[ABS] | k_empty[ABS] | s_full[2] | s_empty[2]; "full" and s_empty are the even CTA's
  __shared__ __align__(8) uint64_t bars[4 * ABS + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(bars);
  auto QF = [&](int i) { return bar0 + 8u * i; };
  auto KF = [&](int i) { return bar0 + 8u * (ABS + i); };
  auto QE = [&](int i) { return bar0 + 8u * (2 * ABS + i); };
  auto KE = [&](int i) { return bar0 + 8u * (3 * ABS + i); };
  auto SF = [&](int i) { return bar0 + 8u * (4 * ABS + i); };
  auto SE = [&](int i) { return bar0 + 8u * (4 * ABS + 2 + i); };
  if (threadIdx.x == 0) {
    for (int i = 0; i < 4 * ABS + 2; ++i) mbar_init(bar0 + 8u * i, 1);
    mbar_init(SE(0), 16); mbar_init(SE(1), 16);                     // epilogue warps of both CTAs
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) { tmem_alloc2((uint32_t)__cvta_generic_to_shared(&tmem_slot), 512); tmem_relinquish2(); }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                               // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  const uint32_t tm = tmem_slot;
  volatile int* abortp = &abort_flag;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0 && lane == 0) {
      // ---- loads of this CTA: its 128 keys and its half of the tile's rows
      const uint64_t normal = l2_policy_normal();
      int issued = 0, g = 0;                                        // heads and key groups so far
      bool ok = true;
      for (int n = 0; ok;) {
        const int kv_row = it.b * a.cache_seq + it.key0, q_row = it.r0 + (int)rank * (it.w >> 1);
        const uint32_t q_half = (uint32_t)q_box_rows(it.bi) * 128u;   // bytes of a 64-dim half of this CTA's Q rows
        for (int h = 0; h < nh; ++h, ++issued) {                    // h: local head index, hgl: head of the model
          const int s = issued % ABS, u = issued / ABS, hgl = h_first + h;
          if (!mbar_wait(QE(s), (u & 1) ^ 1, abortp, status, 21)) { ok = false; break; }
          if (rank == 0) mbar_expect_tx(QF(s), 4u * q_half);
          tma_load_2d_pair(sQ(s), &maps.q[it.bi], hgl * ADH, q_row, QF(s), normal);
          tma_load_2d_pair(sQ(s) + q_half, &maps.q[it.bi], hgl * ADH + 64, q_row, QF(s), normal);
          if (h % group == 0) {
            const int ks = g % ABS, ku = g / ABS, ggl = hgl / group;
            ++g;
            if (!mbar_wait(KE(ks), (ku & 1) ^ 1, abortp, status, 22)) { ok = false; break; }
            if (rank == 0) mbar_expect_tx(KF(ks), 2u * TILE_BYTES);
            tma_load_2d_pair(sK(ks), &maps.k, ggl * ADH, kv_row, KF(ks), normal);
            tma_load_2d_pair(sK(ks) + HALF_BYTES, &maps.k, ggl * ADH + 64, kv_row, KF(ks), normal);
          }
        }
        if (!kStay || !nth_item(p, ++n, rank, it)) break;
      }
      if (*abortp && rank == 0) {
        for (int h = max(0, issued - ABS); h < issued; ++h) {
          const long long t1 = clock64();
          while (!mbar_try_wait(QF(h % ABS), (h / ABS) & 1) && clock64() - t1 < kWaitCycles) {}
        }
      }
    } else if (warp == 1 && rank == 0) {
      const uint32_t el = elect_one();
      bool ok = true;
      int hc = 0, g = -1;                                           // heads so far, current key group
      for (int n = 0; ok;) {
        const uint32_t q_half = (uint32_t)q_box_rows(it.bi) * 128u;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(it.w >> 3) << 17) | ((256u >> 4) << 24);
        for (int h = 0; h < nh; ++h, ++hc) {
          if (h % group == 0) ++g;
          const int s = hc % ABS, u = hc / ABS, ks = g % ABS, ku = g / ABS, sb = hc & 1;
          if (!mbar_wait_warp(QF(s), u & 1, abortp, status, 23)) { ok = false; break; }
          if (h % group == 0 && !mbar_wait_warp(KF(ks), ku & 1, abortp, status, 24)) { ok = false; break; }
          if (!mbar_wait_warp(SE(sb), ((hc >> 1) & 1) ^ 1, abortp, status, 25)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int i = 0; i < ADH / 16; ++i)
            umma2_bf16_e(el, tm + sb * 256, smem_desc_sw128(sK(ks) + (i >> 2) * HALF_BYTES) + 2 * (i & 3),
                         smem_desc_sw128(sQ(s) + (i >> 2) * q_half) + 2 * (i & 3), idesc, i != 0);
          umma2_commit_pair_e(el, QE(s), both);                             // Q stage free
          if ((h + 1) % group == 0 || h + 1 == nh) umma2_commit_pair_e(el, KE(ks), both);        // last head of the group: K stage free
          umma2_commit_pair_e(el, SF(sb), both);
        }
        if (!kStay || !nth_item(p, ++n, rank, it)) break;
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");           // 384 x 168 at launch = 128 x 40 + 256 x 232
    // eight warps, two per TMEM lane quarter: 32 keys (one per lane) x up to 128 of the tile's rows each
    const int quarter = warp & 3, half = (warp - 4) >> 2, etid = (int)threadIdx.x - 128;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const float sc = kLog2e * rsqrtf((float)ADH), inv = 1.f / (float)a.hq;
    const unsigned long long sc2 = pack2(sc, sc);
    bool ok = true;
    int hc = 0;                                                     // heads so far
    for (int n = 0;;) {
      const int w = it.w, r0 = it.r0, nrows = it.nrows, key0 = it.key0;
      const int c_mid = 32 * ((w + 63) >> 6);
      const int c0 = half ? c_mid : 0, nblk = ((half ? w - c_mid : c_mid) + 31) >> 5;      // blocks of 32 rows
      if (kStay && n > 0) {                                         // everybody has read the previous item's, or all stop together
        int stop;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.eq.s32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                     : "=r"(stop) : "r"((int)ok) : "memory");
        if (stop) break;
      }
      // -lse * log2(e) of every head and row (dead rows: -inf, probability 0)
      for (int i = etid; i < w * nh; i += 256) {
        const int r = i / nh, h = i - r * nh;
        const float e = r < nrows ? -__ldcg(a.lse + (size_t)(r0 + r) * a.hq + h_first + h) * kLog2e : -INFINITY;
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(s_lse + 4u * (uint32_t)(h * w + r)), "f"(e) : "memory");
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      unsigned long long acc[64];                                     // packed pairs of neighbouring rows
#pragma unroll
      for (int i = 0; i < 64; ++i) acc[i] = 0ull;                     // (the bits of 0.f are 0)
      for (int h = 0; h < nh && ok; ++h, ++hc) {
        const int sb = hc & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(SF(sb), (hc >> 1) & 1, abortp, status, 26))) { ok = false; break; }   // whole warp or nobody: tcgen05.ld below
        tc_fence_after();
        const uint32_t ts = tm + sb * 256 + lane_base + c0, se = s_lse + 4u * (uint32_t)(h * w + c0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (c >= nblk) break;                                       // uniform across the warp
          uint32_t v[32];
          tmem_ld32(ts + c * 32, v);
          unsigned long long e2[16];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(e2[2 * q]), "=l"(e2[2 * q + 1]) : "r"(se + (uint32_t)(c * 128 + q * 16)) : "memory");
          tmem_ld_wait();
          if (c == nblk - 1) {                                        // the scores are in registers: the buffer may be refilled
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_even_cta(SE(sb));
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float x0, x1;
            unpack2(fma2(pack2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), sc2, e2[i]), x0, x1);
            acc[c * 16 + i] = add2(acc[c * 16 + i], pack2(exp2f(x0), exp2f(x1)));
          }
        }
        if (nblk == 0) {                                              // a tile of 32 rows or fewer: the other half has them all
          __syncwarp();
          if (lane == 0) mbar_arrive_even_cta(SE(sb));
        }
      }
      const int key = key0 + quarter * 32 + lane;
      if (hgs == 1) {
        float* dst = a.abar + (size_t)(r0 + c0) * L + key;            // 32 consecutive keys per store
#pragma unroll
        for (int i = 0; i < 64; ++i) {
          float x0, x1;
          unpack2(acc[i], x0, x1);
          if (ok && key < L && c0 + 2 * i < nrows && 2 * i < nblk * 32) dst[(size_t)(2 * i) * L] = x0 * inv;
          if (ok && key < L && c0 + 2 * i + 1 < nrows && 2 * i + 1 < nblk * 32) dst[(size_t)(2 * i + 1) * L] = x1 * inv;
        }
      } else {
        // [row][128 keys] over the rings: every MMA has read its operands (the last scores have arrived), and so has the
        // peer's part of them (its tensor core took part in the same MMAs)
#pragma unroll
        for (int i = 0; i < 64; ++i) {
          if (2 * i >= nblk * 32) break;
          float x0, x1;
          unpack2(acc[i], x0, x1);
          const uint32_t at = base + (uint32_t)((c0 + 2 * i) * 512 + (quarter * 32 + lane) * 4);
          asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(x0 * inv) : "memory");
          asm volatile("st.shared.f32 [%0], %1;" ::"r"(at + 512u), "f"(x1 * inv) : "memory");
        }
      }
      if (!kStay || !nth_item(p, ++n, rank, it)) break;
    }
  }
  if (hgs > 1) {
    __syncwarp();
    cluster_sync_all();
    if (warp >= 4 && !*abortp) {
      const int r0 = it.r0, nrows = it.nrows, key0 = it.key0;
      // this CTA's share of the tile's rows, a warp a row: the same keys of every pair of the cluster
      const int ra = nrows * hg / hgs, rb = nrows * (hg + 1) / hgs;
      const int key = key0 + 4 * lane;
      const bool vec = (L & 3) == 0 && (reinterpret_cast<uintptr_t>(a.abar) & 15) == 0;
#pragma unroll 2
      for (int r = ra + (warp - 4); r < rb; r += 8) {
        const uint32_t at = base + (uint32_t)(r * 512 + lane * 16);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int g2 = 0; g2 < 4; ++g2) {
          if (g2 < hgs) {
            uint32_t ra2;
            float4 x;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra2) : "r"(at), "r"((uint32_t)(2 * g2) + rank));
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(ra2) : "memory");
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
          }
        }
        float* dst = a.abar + (size_t)(r0 + r) * L + key;
        if (vec && key + 4 <= L) {
          *reinterpret_cast<float4*>(dst) = s;
        } else {
          if (key < L) dst[0] = s.x;
          if (key + 1 < L) dst[1] = s.y;
          if (key + 2 < L) dst[2] = s.z;
          if (key + 3 < L) dst[3] = s.w;
        }
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                               // nobody leaves while the peer may still signal it
  if (warp == 1) { tc_fence_after(); tmem_dealloc2(tm, 512); }
}

}  // namespace

// True if the tcgen05 kernels can take this problem (otherwise the caller uses the mma.sync ones).
bool attention_tc_supported(const AttnArgs& a) {
  return a.dh == ADH && a.hq <= 512 && a.q_rows >= AQ && (long long)a.batch * a.cache_seq >= AKEYS && (a.ldq & 7) == 0 &&
         (reinterpret_cast<uintptr_t>(a.q) & 15) == 0 && (reinterpret_cast<uintptr_t>(a.kc) & 15) == 0 &&
         (reinterpret_cast<uintptr_t>(a.vc) & 15) == 0;
}

// Pairs of SMs that run at the same time when `hgs` of them form a cluster (a cluster stays inside a GPC, whose SM count
// it seldom divides).  Looked up once per device.
static int pairs_at_once(int hgs, int smem) {
  static int known[kMaxDevices][3] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 32;
  int& n = known[dev][hgs >> 1];
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * hgs * 148); cfg.blockDim = dim3(ABAR_THREADS); cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2 * hgs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int clusters = 0;
    (void)cudaFuncSetAttribute(attn_abar_tc<ABAR_GRID>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (cudaOccupancyMaxActiveClusters(&clusters, attn_abar_tc<ABAR_GRID>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); clusters = 32 / hgs; }
    n = clusters > 0 ? clusters * hgs : 1;
  }
  return n;
}

static int expected_rows_per_seq(const AttnArgs& a) {
  const int worst = a.batch * a.max_rows_per_seq, rows = a.expect_rows > 0 && a.expect_rows < worst ? a.expect_rows : worst;
  return ceil_div(rows > 0 ? rows : 1, a.batch);
}

struct AbarCut { int hgs, row_tile, ctas, waves; };
static AbarCut abar_cut(const AttnArgs& a, float* us = nullptr) {
  // How the work is cut: row tiles of 64, 128 or 256 rows (or any multiple of 16, see below), heads shared by 1, 2 or 4 pairs (whole kv groups each); the
  // cheapest by this estimate of waves x time of a CTA (us, measured: a head of a 256-row tile takes 1.8, of a narrow one
  // the loads' 0.5; 6 for set-up, first loads and output; 2 for the meeting).  The row count is an expectation (worst case
  // if there is none): it decides how the work is cut, not what is covered.  Beside other kernels the fewest SMs are best.
  const int kpairs = ceil_div(a.seq_len, 2 * AKEYS), kv_group = a.hq / a.hkv;
  const int rows_seq = expected_rows_per_seq(a), units = ceil_div(rows_seq, 16);
  float best = 1e30f;
  AbarCut cut = {1, 16, 2 * kpairs * a.batch * units, 1};         // (more than 128 heads)
  auto consider = [&](int hgs, int tiles, int tile) {
    const int nh = a.hq / hgs, w = 16 * ceil_div(units, tiles);
    if (tile * nh > ABAR_MAX_ROWS * 32) return;                     // the staged log-sum-exp
    const int at_once = a.pairs > 0 ? a.pairs : pairs_at_once(hgs, kAbarSmem), waves = ceil_div(kpairs * a.batch * tiles * hgs, at_once);
    const float per_head = 0.3f + 1.5f * (float)w / 256.f;
    const float est = (float)waves * ((float)nh * (per_head > 0.5f ? per_head : 0.5f) + 6.f + (hgs > 1 ? 2.f : 0.f));
    if (est < best) { best = est; cut = {hgs, tile, 2 * kpairs * a.batch * tiles * hgs, waves}; }
  };
  const int most_hgs = a.beside || a.pairs > 0 ? 1 : 4;
  auto shared = [&](int hgs) { return a.hq % hgs == 0 && (a.hq / hgs) % kv_group == 0; };
  for (int hgs = 1; hgs <= most_hgs; hgs *= 2)
    for (int tile = 256; tile >= 64 && shared(hgs); tile /= 2) consider(hgs, ceil_div(rows_seq, tile), tile);
  // Where that takes several waves, any number of tiles between: 976 rows of four sequences x 1536 keys took three waves of half of 28
  // heads each, and six tiles of 176 rows take two (four layers 5823 -> 5793 us; 1012 rows x 1500, 32 heads, three layers 1342 -> 1338).  A
  // tile has room for sixteen rows a sequence more than are expected, so that a few more do not make another tile.
  if (cut.waves > 1 && a.pairs == 0 && !a.beside)
    for (int hgs = 1; hgs <= most_hgs; hgs *= 2)
      for (int tiles = ceil_div(units, 16); tiles <= ceil_div(units, 4) && shared(hgs); ++tiles) {
        const int tile = 16 * ceil_div(units + 1, tiles);
        consider(hgs, tiles, tile < ABAR_MAX_ROWS ? tile : ABAR_MAX_ROWS);
      }
  if (us) *us = best;
  return cut;
}

// Pairs on which the pass of a layer keeps up with a layer of layer_us when it runs beside the layer's other kernels, which
// then have only the other SMs; 0 if that costs more than the pass on the whole GPU between them.  Beside GEMMs a head takes
// 1.5 times as long as alone (2.7 us a 256-row tile; with fewer pairs the layers waited for their passes: 489 rows x 32 layers
// 8860 us on two pairs, 8250 on three, 8360 between the other kernels).
int attention_abar_pairs(const AttnArgs& a, float layer_us) {
  float alone = 0.f, us = 0.f;
  AttnArgs t = a;
  t.beside = 0; t.pairs = 0;
  abar_cut(t, &alone);
  const int half = sm_count_current() / 2;
  for (t.pairs = 1; t.pairs <= half / 8; ++t.pairs) {
    abar_cut(t, &us);
    if (us * 1.6f > layer_us) continue;
    return 1.15f * layer_us * (float)t.pairs / (float)half < alone + 2.f ? t.pairs : 0;
  }
  return 0;
}

// SMs the probabilities kernel is expected to hold.
int attention_abar_sms(const AttnArgs& a) {
  if (!a.portable && attention_tc_supported(a)) return abar_cut(a).ctas;
  return ceil_div(ceil_div(a.seq_len, 64) * ceil_div(expected_rows_per_seq(a), 64) * a.batch, 4);     // (about four of its CTAs share an SM)
}

int launch_attention_tc(const AttnArgs& a, cudaStream_t st, int* status) {
  const int smem_fwd = 6 * TILE_BYTES + 1024;
  const uint64_t kv_cols = (uint64_t)a.hkv * a.dh, kv_rows = (uint64_t)a.batch * a.cache_seq;
  const int sms = sm_count_current();
  if (!status) D2C_CUDA_OK(cudaGetSymbolAddress(reinterpret_cast<void**>(&status), g_attn_status));
  // A query tile holds the rows of all query heads of a K/V head, (row, head) by (row, head), as many whole rows as there is room for: 18
  // rows of seven heads, where a head's own rows filled their last tile only in part.  Forward alone, a head's rows / a group's, us, 28 heads
  // over 4: 260 rows of eight sequences x 700 keys 48.6 / 33.6, 147 of four x 1187 24.5 / 21.2, 976 of four x 1536 100.4 / 93.6.
  // Not where a head's tiles by themselves are few enough for as many CTAs to share their keys: the tiles then have fewer rows to finish with
  // (four layers, 18 rows x 600, 28 heads over 4, 644 / 630 us; 28 rows x 1390 671 / 659).
  const int rows_seq = expected_rows_per_seq(a), key_tiles = ceil_div(a.seq_len, AKEYS);
  // Few tiles (expected): 2 to 4 CTAs share a tile's keys while all of them still run at once.  Four only
  // for many key tiles: measured alone at 32 heads (us, 1 / 2 / 3 / 4 CTAs) 768 keys 20.4 / 18.4 / 16.4 / 17.3,
  // 2048 keys 36.8 / 27.6 / 24.6 / 22.5, 4096 keys 64.4 / 43.0 / 36.8 / 31.7.
  auto splits_of = [&](int units) {
    int splits = 1;
    for (int s = 2; s <= kMaxSplits; ++s)
      if (s * units <= sms - 16 && key_tiles >= (s == 4 ? 16 : s + 1)) splits = s;
    return splits;
  };
  const int solo = splits_of(ceil_div(rows_seq, AQ) * a.hq * a.batch), packed = AQ / (a.hq / a.hkv);
  const bool pack = packed > 0 && (solo == 1 || solo < splits_of(ceil_div(rows_seq, packed) * a.hkv * a.batch));      // (a tile has no place for more than 128 heads)
  const int group = pack ? a.hq / a.hkv : 1, heads = a.hq / group, tile_rows = AQ / group;
  AttnTcParams p{a, status, sms, 1, 1, 128, 0, group, heads, a.hq / a.hkv / group, tile_rows, 0, 0};
  if (a.which != 2) {
    static PerDevice attr_set;
    if (attr_set.first()) {
      for (auto* k : {attn_fwd_tc<false, false, false>, attn_fwd_tc<false, true, false>, attn_fwd_tc<true, false, false>, attn_fwd_tc<true, true, false>,
                      attn_fwd_tc<true, false, true>, attn_fwd_tc<true, true, true>, attn_fwd_tc<false, false, true>, attn_fwd_tc<false, true, true>})
        D2C_CUDA_OK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_fwd));
    }
    struct Maps { CUtensorMap q, k, v; } fresh, *m = &fresh;
    bool made = false;
    if (a.cache[0]) {
      m = reinterpret_cast<Maps*>(a.cache[0]->maps);
      made = a.cache[0]->same(a.q, a.kc, a.vc, a.q_rows, a.hq, a.ldq, (long long)kv_rows, (long long)kv_cols, 3 + 8 * group);
    }
    if (!made) {
      // (one head a tile: rows by columns; as boxes of (row, head) they come in 0.25 us later)
      int rc = group == 1 ? make_bf16_map(&m->q, a.q, (uint64_t)a.q_rows, (uint64_t)a.hq * a.dh, (uint64_t)a.ldq, AQ)
                          : make_bf16_head_map(&m->q, a.q, (uint64_t)a.q_rows, (uint64_t)a.hq, (uint64_t)a.ldq, (uint32_t)tile_rows, (uint32_t)group);
      if (rc == D2C_OK) rc = make_bf16_map(&m->k, a.kc, kv_rows, kv_cols, kv_cols, 128);
      if (rc == D2C_OK) rc = make_bf16_map(&m->v, a.vc, kv_rows, kv_cols, kv_cols, 128);
      if (rc != D2C_OK) { if (a.cache[0]) a.cache[0]->forget(); return rc; }
    }
    const int units = ceil_div(rows_seq, tile_rows) * heads * a.batch;
    p.splits = splits_of(units);
    cudaLaunchConfig_t cfg = {};
    const int xtiles = ceil_div(a.max_rows_per_seq, tile_rows);
    // (as many CTAs as there can be items: one a tile up to the SMs, one a pair of tiles beyond)
    const int most = heads * a.batch * ((xtiles + 1) / 2), single = heads * a.batch * xtiles < sms ? heads * a.batch * xtiles : sms;
    // With shared keys there are places for all tiles where more than half of them are expected (two layers of d 512, all of 521 rows, 128 us,
    // with places for half 134) or where the CTAs without rows are at most two waves behind the others; beyond, clusters for half of the tiles,
    // which take two each where that is not enough.  Places for half / all, us: four layers, 28 heads over 4, 60 rows of 350 positions (252
    // CTAs in all) 649 / 646, 500 (336) 645 / 634, 18 of 600 (420) 624 / 618, 32 heads 18 of 400 (384) 576 / 566; two of d 512, 100 rows of each
    // of eight sequences of 300 (192) 144.0 / 140.5; but 32 heads 18 of 600 (480) 574 / 582, 28 heads 60 of 1024 (672) 644 / 649, 28 of 1390
    // (924) 638 / 646; 32 layers at 80 of 768 (576) 3775 / 3810.
    const bool one = 2 * ceil_div(rows_seq, tile_rows) > xtiles || (long long)p.splits * heads * a.batch * xtiles <= 3 * sms;
    const int clusters = one ? xtiles : (xtiles + 1) / 2;
    if ((long long)clusters * a.batch > 65535) p.splits = 1;      // (tiles of a few rows, of many long sequences: the grid has no room for their places)
    const int pairs = ceil_div(ceil_div(rows_seq, tile_rows), 2) * heads * a.batch;      // (expected; where none are to be split, looking for them costs 0.4 us)
    p.split_last = units > sms && pairs > sms && pairs % sms > 0 && 2 * (pairs % sms) <= sms;
    // By place where all places run at once: two layers of d 512, all rows of eight sequences of 300, 179.7 -> 177.8 us a step.  And where there
    // are two at most and one tile is expected: no CTA has a pair then, and finding its number took each of them longer than the empty ones
    // between do.  Four layers of d 4096, in turn / by place: 100 rows of five sequences of 215 positions 666 / 659 us, forward alone 21.7 / 20.5;
    // 160 of eight x 215, 256 of three x 250, 400 of four x 256 and 800 of eight x 140 no difference.
    const bool by_place = p.splits == 1 && (single < sms || (xtiles <= 2 && rows_seq <= tile_rows));
    p.places = p.splits > 1 ? clusters : by_place ? xtiles : 0;
    cfg.gridDim = p.splits > 1 ? dim3(p.splits, heads, clusters * a.batch) : by_place ? dim3(heads * a.batch * xtiles) : dim3((most > single ? most : single) + (p.split_last ? sms / 2 : 0));
    cfg.blockDim = dim3(FWD_THREADS); cfg.dynamicSmemBytes = smem_fwd; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = p.splits; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = p.splits > 1 ? 2 : 1;
    auto* kernel = group > 1 ? attn_fwd_tc<false, true, false> : attn_fwd_tc<false, false, false>;
    if (by_place) kernel = group > 1 ? attn_fwd_tc<false, true, true> : attn_fwd_tc<false, false, true>;
    else if (p.splits > 1 && one) kernel = group > 1 ? attn_fwd_tc<true, true, true> : attn_fwd_tc<true, false, true>;
    else if (p.splits > 1) kernel = group > 1 ? attn_fwd_tc<true, true, false> : attn_fwd_tc<true, false, false>;
    D2C_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, m->q, m->k, m->v, p));
    count_launch(1);
  }
  if (!a.abar || a.which == 1) return D2C_OK;
  static PerDevice attr_set;
  if (attr_set.first()) {
    for (auto* k : {attn_abar_tc<ABAR_GRID>, attn_abar_tc<ABAR_IN_TURN>, attn_abar_tc<ABAR_STAY>})
      D2C_CUDA_OK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kAbarSmem));
  }
  const AbarCut cut = abar_cut(a);
  p.head_groups = cut.hgs; p.row_tile = cut.row_tile; p.pairs = a.pairs;
  AbarMaps fresh, *m = &fresh;
  static_assert(sizeof(AbarMaps) <= sizeof(MapCache::maps), "the cache holds one launch's maps");
  bool made = false;
  if (a.cache[1]) {
    m = reinterpret_cast<AbarMaps*>(a.cache[1]->maps);
    made = a.cache[1]->same(a.q, a.kc, nullptr, a.q_rows, a.hq, a.ldq, (long long)kv_rows, (long long)kv_cols, 4);
  }
  if (!made) {
    int rc = make_bf16_map(&m->k, a.kc, kv_rows, kv_cols, kv_cols, 128);
    for (int i = 0; i < N_QBOX && rc == D2C_OK; ++i)
      rc = make_bf16_map(&m->q[i], a.q, (uint64_t)a.q_rows, (uint64_t)a.hq * a.dh, (uint64_t)a.ldq, (uint32_t)q_box_rows(i));
    if (rc != D2C_OK) { if (a.cache[1]) a.cache[1]->forget(); return rc; }
  }
  cudaLaunchConfig_t cfg = {};
  // The live items are numbered in turn, as in the forward, where there is room for twice as many tiles of rows as are expected, or more, and
  // so for more than two CTAs an SM that would find nothing to do.  us, by place / in turn: 300 rows of five sequences x 3071 keys 100.5 / 95.8,
  // 147 of four x 1187 32.4 / 31.1, 420 of three x 1100 38.3 / 37.8.  Finding its number takes a cluster up to 0.9 us: with fewer tiles than that
  // 260 rows of eight x 700 41.8 / 42.7.  Two to eight sequences of 300 to 2048 positions, 4 to 150 rows each, 4, 28 and 32 heads: with up to two
  // empty CTAs an SM 1.5 more (8 rows of two x 701, 4 heads, 14.7 / 15.8) to 1.8 less (28 heads, 160 of eight x 701 20.0 / 18.1), beyond
  // 0.3 to 9 less (28 heads, 32 rows of eight x 2048 36.5 / 30.5), but for 300 rows of two x 2048, 28.8 / 30.4.
  const int xs = 2 * p.head_groups * ceil_div(a.seq_len, 2 * AKEYS), worst_tiles = ceil_div(a.max_rows_per_seq, p.row_tile);
  const int empty = xs * a.batch * (worst_tiles - ceil_div(rows_seq, p.row_tile));
  const bool in_turn = a.batch > 1 && worst_tiles >= 2 * ceil_div(rows_seq, p.row_tile) && empty > 2 * sms;
  cfg.gridDim = p.pairs > 0 ? dim3(2 * p.pairs) : (in_turn ? dim3(xs * worst_tiles * a.batch) : dim3(xs, worst_tiles, a.batch));
  cfg.blockDim = dim3(ABAR_THREADS); cfg.dynamicSmemBytes = kAbarSmem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2 * p.head_groups; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  D2C_CUDA_OK(cudaLaunchKernelEx(&cfg, p.pairs > 0 ? attn_abar_tc<ABAR_STAY> : in_turn ? attn_abar_tc<ABAR_IN_TURN> : attn_abar_tc<ABAR_GRID>, *m, p));
  count_launch(1);
  return D2C_OK;
}

}  // namespace d2c

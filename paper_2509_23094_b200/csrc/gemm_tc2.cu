// Two-SM tcgen05 GEMM (cta_group::2) of the projections, with the step's fused epilogues.
//
//   C[t][f] = sum_k A[t][k] * W[f][k]      A: activations (tokens x K), W: weights (features x K), both K-major bf16
//
// The weights are the M operand and the tokens the N operand.  A cluster of two CTAs (two SMs) owns 256 weight rows
// (a block: CTA r holds 128 of them, its TMEM lanes) and up to 256 tokens (the accumulator's columns, half of whose
// rows each CTA brings in): tcgen05.mma.cta_group::2, M = 256, K = 16, N any multiple of 16.  The selected-row count
// of a step is arbitrary and the model's widths are multiples of 128, so this way round nothing is computed for
// padding: with the tokens on M, 831 rows ran as 1024, 588 as 768 and 81 as 128.
//
// Work.  The tokens are cut into TT = ceil(n / 256) tiles of almost equal width.  Whole (block, token tile) items are
// handed out in waves, token tile fastest: clusters running together share a weight block, which crosses from HBM
// once.  What does not fill a wave (all of it, when few rows are live) is shared: its run of pipeline stages is cut
// into equal parts, one per cluster (stream-K), or, with up to eight token tiles, one per group of TT clusters that
// walk the same weights for a token tile each.  Parts of a split item are parked as fp32 in scratch; its contributors
// meet at a counter and each adds the parts (in part order: deterministic) and finishes the epilogue for its own share
// of the (16 tokens x 32 lanes) cells.  A cluster works on its parts before its whole items, so that the meeting and
// the adding hide behind the next item's MMAs; a cluster without whole items leaves its own part in TMEM.
//
// Per CTA: warp 0 loads (TMA; warp 10 the first activations), warp 1 of the even CTA issues the MMAs, warps 2-9 run the
// epilogue, two per TMEM lane quarter on half of the token columns each.  A pipeline stage holds two 64-wide k-blocks, so
// that a barrier test and a commit serve eight MMAs (stages of one k-block: 333 rows of a small model 126.0 -> 128.3 us, the large
// steps no different).
// TMA loads of both CTAs signal the even CTA's mbarrier (no multicast load); stage release and accumulator hand-over
// reach both CTAs through multicast tcgen05.commit.
//
// Epilogue.  TMEM is read in the 16x256b shape: a thread holds two neighbouring tokens of features T/4 and T/4 + 8, the
// register layout of an 8x8 matrix fragment, so a rounded pair of tokens is transposed to [token][feature] by
// stmatrix.trans into 2 KB of shared memory per warp and leaves in 16-byte stores; the residual comes in the same way
// through ldmatrix.trans.  Work that pairs features (SwiGLU's gate and up, the halves of a rotary pair) has the two in
// different warps: the warps of a pair swap half of their tokens through the same 2 KB, register for register, and each
// finishes the other half.  (Weight boxes of 16 rows, which put partners 16 lanes apart and need no swap, cost 0.95 us
// a stage instead of 0.62: eight TMA boxes per k-block are too many.)
#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tc2_work.cuh"

namespace d2c {
// No more clusters than there are token tiles times shares of three stages, or 64-token tiles.
static long long share_clusters(long long blocks, long long rows, int K) { return blocks * ((rows + 255) / 256) * ceil_div(ceil_div(K, 128), 3); }
static long long narrow_clusters(long long blocks, long long rows) { return blocks * ((rows + 63) / 64); }
long long gemm_tc2_clusters(long long blocks, long long rows, int K) {
  const long long shares = share_clusters(blocks, rows, K), narrow = narrow_clusters(blocks, rows);
  return narrow > shares ? narrow : shares;
}
int gemm_tc2_ctas(const GemmArgs& g, GemmEpilogue epi, bool narrow_tiles) {
  const long long blocks = ceil_div(g.N, epi == EPI_SWIGLU ? 128 : 256);
  const long long shares = share_clusters(blocks, g.max_rows, g.K), all = narrow_clusters(blocks, g.max_rows);
  const long long narrow = g.narrow_pairs > 0 && g.narrow_pairs < all ? g.narrow_pairs : all;
  const long long most = narrow_tiles && narrow > shares ? narrow : shares;
  const int fit = g.max_pairs > 0 && g.max_pairs < sm_count_current() / 2 ? g.max_pairs : sm_count_current() / 2;
  return 2 * (int)(most < fit ? most : fit);
}
// How the product is cut depends on this and on the row count.  A block's 256 weight rows make 128 or 256 output features.
WorkShape gemm_tc2_shape(const GemmArgs& g, GemmEpilogue epi) {
  return {ceil_div(g.N, epi == EPI_SWIGLU ? 128 : 256), g.K, gemm_tc2_ctas(g, epi) / 2, g.sk_partials && g.sk_counters && gemm_tc2_ctas(g, epi) <= kPairCounters ? g.sk_max_tiles : 0};
}

namespace {

constexpr int EPI_WARPS = 8;
constexpr int TOKEN_WARP = 2 + EPI_WARPS;
constexpr int TC_THREADS = 32 * (TOKEN_WARP + 1);
constexpr int W_BYTES = 128 * TK * 2;             // 16 KB: this CTA's weight rows of one k-block
constexpr int NST_MAX = 6;
constexpr int RING_BYTES = 200 * 1024;
constexpr int EPI_STAGE_BYTES = 2048;             // per epilogue warp: 32 tokens x 32 features of bf16
constexpr int N_BOXES = 6;                        // heights of the token boxes (tokens per CTA, k-block)
constexpr int SLOT_F4 = 128 * MAX_TOK / 4;        // float4 elements of one scratch slot: [unit][quarter][4][lane]

__host__ __device__ constexpr int box_rows(int i) { return i == 0 ? 16 : i == 1 ? 32 : i == 2 ? 48 : i == 3 ? 64 : i == 4 ? 96 : 128; }

__device__ int g_tc_status[4];

__device__ __forceinline__ uint32_t bf16x2_bits(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float2 bf16x2_floats(uint32_t v) {
  return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&v));
}
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 32 accumulator columns of 16 TMEM lanes: v[4 j + 2 b + e] = column 8 j + 2 (T % 4) + e of lane T / 4 + 8 b.
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                 "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

struct Tc2Maps { CUtensorMap w, w2, tok[N_BOXES]; };
struct Tc2Params { GemmArgs g; WorkShape shape; int* status; };

// A cluster's part of a split item: the item, the first group that holds some of it, the number of parts, this
// cluster's place among them, and the cells (16 tokens x the lanes that finish features together) that it finishes.
struct Part { int nb, tile, g0, parts, mine, a0, a1; };

// ------------------------------------------------------------------------------------------- epilogue arithmetic
// An epilogue warp works on 32 tokens of its 32 TMEM lanes at a time: v[16 h + 4 j + 2 b + e] is token 8 j + 2 (T % 4) + e
// of lane 16 h + 8 b + T / 4.  Where features are paired it then holds v[0..15] of the lower and v[16..31] of the upper
// partner, both [8 h + 4 j + 2 b + e], for the 16 tokens that it finishes.
struct EpiTile {
  const GemmArgs& g;
  int t0, n;                           // first token of the tile, end of the tokens to store
  int lane, f;                         // f: the warp's first feature (the lower partners', where paired)
  uint32_t stage, stage_base;          // the warp's shared-memory buffer, the first warp's
  const float* scale;                  // per token of the tile: factor of the folded RMSNorm (null: none)
  const int* pos; const int* crow;     // per token (QKV): position, row of the K/V cache
  uint32_t half_stage; int quarter, stile;      // LM head: the four warps' buffers, this warp's lane quarter, index of the 128 features
  // 16-byte piece pc of row tk of the staged tile (rows of 64 bytes, swizzled over the banks)
  __device__ uint32_t at4(int tk, int pc) const { return stage + (uint32_t)(tk * 64 + ((pc ^ ((tk >> 1) & 3)) << 4)); }
};

// What the arithmetic of a chunk needs from memory, requested a chunk ahead.
template <int EPI> struct EpiPre {
  __device__ void load(const EpiTile&, int) {}
};
template <> struct EpiPre<EPI_RESIDUAL> {
  uint4 old[4];
  __device__ void load(const EpiTile& e, int tk0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = e.t0 + tk0 + 8 * i + (e.lane >> 2), col = e.f + 8 * (e.lane & 3);
      old[i] = (row < e.n && col < e.g.N) ? __ldcg(reinterpret_cast<const uint4*>(e.g.C + (size_t)row * e.g.ldc + col)) : make_uint4(0, 0, 0, 0);
    }
  }
};
template <> struct EpiPre<EPI_QKV_ROPE> {
  float2 cs[16];                       // [h][j][b][e], tokens tk0 .. tk0 + 15
  __device__ void load(const EpiTile& e, int tk0) {
    const int dh = e.g.q_dh, half = dh >> 1, head = e.f / dh, t = e.f - head * dh + (e.lane >> 2);
    if (head >= e.g.q_hq + e.g.q_hkv) return;                // V: nothing to rotate
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2* row = e.g.q_rope + (size_t)e.pos[tk0 + 8 * j + 2 * (e.lane & 3) + k] * half + t;
#pragma unroll
        for (int r = 0; r < 4; ++r) cs[8 * (r >> 1) + 4 * j + 2 * (r & 1) + k] = __ldg(row + 8 * r);
      }
  }
};

// Rounds v to bf16 and leaves it staged as [32 tokens][32 lanes].
__device__ __forceinline__ void stage_rows(const EpiTile& e, const float (&v)[32]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    stmatrix_x4_trans(e.at4(8 * j + (e.lane & 7), e.lane >> 3), bf16x2_bits(v[4 * j], v[4 * j + 1]), bf16x2_bits(v[4 * j + 2], v[4 * j + 3]),
                      bf16x2_bits(v[16 + 4 * j], v[16 + 4 * j + 1]), bf16x2_bits(v[16 + 4 * j + 2], v[16 + 4 * j + 3]));
  __syncwarp();
}
// Copies the staged rows to out[token][f + ...].
__device__ __forceinline__ void store_rows(const EpiTile& e, bf16* out, int tk0) {
  const GemmArgs& g = e.g;
  const int pc = e.lane & 3, col = e.f + 8 * pc;
  const bool vec = ((g.ldc | g.N) & 7) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int tk = 8 * i + (e.lane >> 2), row = e.t0 + tk0 + tk;
    const uint4 w = lds128(e.at4(tk, pc));
    if (row >= e.n || col >= g.N) continue;
    bf16* dst = out + (size_t)row * g.ldc + col;
    if (vec) {
      *reinterpret_cast<uint4*>(dst) = w;
    } else {
      const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&x[q]);
        if (col + 2 * q < g.N) dst[2 * q] = __low2bfloat16(h);
        if (col + 2 * q + 1 < g.N) dst[2 * q + 1] = __high2bfloat16(h);
      }
    }
  }
  __syncwarp();                        // the buffer may be filled again
}

// Tokens tk0 .. of the tile (32 of them; 16 where features are paired); asks for the data of the next chunk's as soon as
// `pre` has been used.
template <int EPI>
__device__ __forceinline__ void finish(const EpiTile& e, float (&v)[32], int tk0, EpiPre<EPI>& pre, bool more) {
  const GemmArgs& g = e.g;
  const int fr = e.lane >> 2, tc = 2 * (e.lane & 3);          // this thread's first lane row and token column
  constexpr bool pairs = EPI == EPI_SWIGLU || EPI == EPI_QKV_ROPE;
  if (e.scale) {
#pragma unroll
    for (int j = 0; j < (pairs ? 2 : 4); ++j) {
      const float2 s = *reinterpret_cast<const float2*>(e.scale + tk0 + 8 * j + tc);
#pragma unroll
      for (int r = 0; r < (pairs ? 8 : 4); ++r) {
        const int i = (pairs ? 8 : 16) * (r >> 1) + 4 * j + 2 * (r & 1);
        v[i] *= s.x; v[i + 1] *= s.y;
      }
    }
  }
  if constexpr (EPI == EPI_STORE) {
    if (g.bias) {
      float add[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) { const int f = e.f + 8 * r + fr; add[r] = f < g.N ? __bfloat162float(g.bias[f]) : 0.f; }
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] += add[2 * (i >> 4) + ((i >> 1) & 1)];
    }
    stage_rows(e, v);
    store_rows(e, g.C, tk0);
  } else if constexpr (EPI == EPI_RESIDUAL) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sts128(e.at4(8 * i + (e.lane >> 2), e.lane & 3), pre.old[i]);
    if (more) pre.load(e, tk0 + 32);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t o[4];
      ldmatrix_x4_trans(e.at4(8 * j + (e.lane & 7), e.lane >> 3), o[0], o[1], o[2], o[3]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float2 x = bf16x2_floats(o[r]);
        const int i = 16 * (r >> 1) + 4 * j + 2 * (r & 1);
        v[i] += x.x; v[i + 1] += x.y;
      }
    }
    __syncwarp();
    stage_rows(e, v);
    store_rows(e, g.C, tk0);
    if (g.nx_out) {
      // the next RMSNorm, folded: x * gain for the next GEMM and the sum of squares of the row's 32 features, both
      // from the stored bf16 x
      float gain[4], sq[8];
#pragma unroll
      for (int r = 0; r < 4; ++r) { const int f = e.f + 8 * r + fr; gain[r] = f < g.N ? __bfloat162float(g.nx_gain[f]) : 0.f; }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sq[2 * j] = sq[2 * j + 1] = 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int i = 16 * (r >> 1) + 4 * j + 2 * (r & 1);
          const float2 x = bf16x2_floats(bf16x2_bits(v[i], v[i + 1]));
          if (e.f + 8 * r + fr < g.N) { sq[2 * j] += x.x * x.x; sq[2 * j + 1] += x.y * x.y; }
          v[i] = x.x * gain[r]; v[i + 1] = x.y * gain[r];
        }
      }
      // sums over the eight lanes of a token; each step also halves the tokens a lane carries
      int item = 0;
#pragma unroll
      for (int h = 4; h >= 1; h >>= 1) {
        const bool up = e.lane & (4 * h);
#pragma unroll
        for (int i = 0; i < h; ++i) {
          const float keep = up ? sq[i + h] : sq[i], give = up ? sq[i] : sq[i + h];
          sq[i] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
        }
        item += up ? h : 0;
      }
      const int row = e.t0 + tk0 + 8 * (item >> 1) + tc + (item & 1);
      if (g.nx_ssq && row < e.n && e.f < g.N) g.nx_ssq[(size_t)row * (size_t)(g.N >> 5) + (size_t)(e.f >> 5)] = sq[0];
      stage_rows(e, v);
      store_rows(e, g.nx_out, tk0);
    }
  } else if constexpr (EPI == EPI_SWIGLU) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float hx = 0.5f * v[i];                           // silu(x) = h tanh(h) + h, h = x / 2: one MUFU op
      v[i] = fmaf(hx, tanh_fast(hx), hx) * v[16 + i];
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
      stmatrix_x4_trans(e.at4(8 * j + (e.lane & 7), e.lane >> 3), bf16x2_bits(v[4 * j], v[4 * j + 1]), bf16x2_bits(v[4 * j + 2], v[4 * j + 3]),
                        bf16x2_bits(v[8 + 4 * j], v[8 + 4 * j + 1]), bf16x2_bits(v[8 + 4 * j + 2], v[8 + 4 * j + 3]));
    __syncwarp();
    const int pc = e.lane & 3, col = e.f + 8 * pc;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int tk = 8 * i + (e.lane >> 2), row = e.t0 + tk0 + tk;
      const uint4 w = lds128(e.at4(tk, pc));
      if (row < e.n && col < g.N) *reinterpret_cast<uint4*>(g.C + (size_t)row * g.ldc + col) = w;
    }
    __syncwarp();
  } else if constexpr (EPI == EPI_LMSTATS) {
    // Per token over the CTA's 128 features: maximum, its lowest index, sum of exp(x - max).  First over this warp's 32
    // lanes, then over the four warps through their buffers.  Features past the end count as -inf, which adds nothing; a
    // logit that is not a number is no maximum but makes the sum, and with it the confidence, not a number.
    float mx[8], sum[8];
    int arg[8];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const bool ok = e.f + 8 * r + fr < g.N;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int i = 16 * (r >> 1) + 4 * (t >> 1) + 2 * (r & 1) + (t & 1);
        if (!ok) v[i] = -INFINITY;
      }
    }
    if (g.logits) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int row = e.t0 + tk0 + 8 * (t >> 1) + tc + (t & 1), f = e.f + 8 * r + fr;
          if (row < e.n && f < g.N) g.logits[(size_t)row * g.N + f] = v[16 * (r >> 1) + 4 * (t >> 1) + 2 * (r & 1) + (t & 1)];
        }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i0 = 4 * (t >> 1) + (t & 1);
      mx[t] = fmaxf(fmaxf(v[i0], v[i0 + 2]), fmaxf(v[i0 + 16], v[i0 + 18]));
#pragma unroll
      for (int s = 4; s <= 16; s <<= 1) mx[t] = fmaxf(mx[t], __shfl_xor_sync(0xffffffffu, mx[t], s));
      arg[t] = 0x7fffffff; sum[t] = 0.f;
#pragma unroll
      for (int r = 3; r >= 0; --r) {                          // (the lowest feature wins)
        const float x = v[i0 + 16 * (r >> 1) + 2 * (r & 1)];
        if (x == mx[t] && e.f + 8 * r + fr < g.N) arg[t] = e.f + 8 * r + fr;
        sum[t] += x == -INFINITY ? 0.f : __expf(x - mx[t]);
      }
    }
    int item = 0;                                              // each step also halves the tokens a lane carries
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
      const bool up = e.lane & (4 * h);
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const float ks = up ? sum[i + h] : sum[i], gs = up ? sum[i] : sum[i + h];
        const int ka = up ? arg[i + h] : arg[i], ga = up ? arg[i] : arg[i + h];
        mx[i] = up ? mx[i + h] : mx[i];
        sum[i] = ks + __shfl_xor_sync(0xffffffffu, gs, 4 * h);
        arg[i] = min(ka, __shfl_xor_sync(0xffffffffu, ga, 4 * h));
      }
      item += up ? h : 0;
    }
    const int tok = 8 * (item >> 1) + tc + (item & 1);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(e.stage + (uint32_t)tok * 16u), "r"(__float_as_uint(mx[0])), "r"(__float_as_uint(sum[0])),
                 "r"((uint32_t)arg[0]), "r"(0u) : "memory");
    const int bar = 2 + (int)((e.half_stage - e.stage_base) / (4u * EPI_STAGE_BYTES));
    asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
    if (e.lane < 8) {
      const int tk = e.quarter * 8 + e.lane, row = e.t0 + tk0 + tk;
      float m = -INFINITY, s = 0.f;
      int am = 0x7fffffff;
      uint4 p[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { p[q] = lds128(e.half_stage + (uint32_t)((q + 2) & 3) * EPI_STAGE_BYTES + (uint32_t)tk * 16u); m = fmaxf(m, __uint_as_float(p[q].x)); }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float pm = __uint_as_float(p[q].x);
        if (pm == m) am = min(am, (int)p[q].z);
        s = fmaf(__uint_as_float(p[q].y), pm == -INFINITY ? 1.f : __expf(pm - m), s);
      }
      if (row < e.n && e.stile < g.n_tiles) {
        const size_t o = (size_t)row * g.n_tiles + e.stile;
        g.st_max[o] = m; g.st_sum[o] = s; g.st_arg[o] = am;
      }
    }
    asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
  } else {
    // Bias, rotary embedding of Q and K at the token's position, Q to the activation buffer, K and V to their cache row
    const int dh = g.q_dh, half = dh >> 1, head = e.f / dh, t = e.f - head * dh;
    const bool is_q = head < g.q_hq, is_k = !is_q && head < g.q_hq + g.q_hkv;
    if (g.bias && e.f < g.N) {
      float lo[4], hi[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) { lo[r] = __bfloat162float(g.bias[e.f + 8 * r + fr]); hi[r] = __bfloat162float(g.bias[e.f + half + 8 * r + fr]); }
#pragma unroll
      for (int i = 0; i < 16; ++i) { const int r = 2 * (i >> 3) + ((i >> 1) & 1); v[i] += lo[r]; v[16 + i] += hi[r]; }
    }
    if (is_q || is_k) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        // the projection result is rounded to bf16 before the rotation, as the unfused path stores it
        const float l = __bfloat162float(__float2bfloat16_rn(v[i])), h = __bfloat162float(__float2bfloat16_rn(v[16 + i]));
        v[i] = l * pre.cs[i].x - h * pre.cs[i].y;
        v[16 + i] = h * pre.cs[i].x + l * pre.cs[i].y;
      }
    }
    if (more) pre.load(e, tk0 + 32);
#pragma unroll
    for (int p = 0; p < 2; ++p)                               // rows 0..15 of the buffer: lower partners, 16..31: upper
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float* x = v + 16 * p + 4 * j;
        stmatrix_x4_trans(e.at4(16 * p + 8 * j + (e.lane & 7), e.lane >> 3), bf16x2_bits(x[0], x[1]), bf16x2_bits(x[2], x[3]),
                          bf16x2_bits(x[8], x[9]), bf16x2_bits(x[10], x[11]));
      }
    __syncwarp();
    const int pc = e.lane & 3, hh = head - g.q_hq - (is_k ? 0 : g.q_hkv);
    bf16* base = (is_q ? g.C + (size_t)head * dh : (is_k ? g.q_kc : g.q_vc) + (size_t)hh * dh) + t + 8 * pc;
    const size_t ld = is_q ? (size_t)g.ldc : (size_t)(g.q_hkv * dh);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int tk = 8 * i + (e.lane >> 2), row = e.t0 + tk0 + tk;
      const uint4 lo = lds128(e.at4(tk, pc)), hi = lds128(e.at4(16 + tk, pc));
      if (row < e.n && e.f < g.N) {
        bf16* dst = base + (size_t)(is_q ? row : e.crow[tk0 + tk]) * ld;
        *reinterpret_cast<uint4*>(dst) = lo;
        *reinterpret_cast<uint4*>(dst + half) = hi;
      }
    }
    __syncwarp();
  }
}

template <int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1)
gemm_tc2_kernel(const __grid_constant__ Tc2Maps maps, const Tc2Params p) {
  // Everything that does not read a predecessor's results (barriers, TMEM, descriptor prefetch) runs before
  // the wait on the preceding kernel, so it overlaps that kernel's tail.
  // The LM head lets its successor launch only when its loads are requested: those CTAs would wait on the SMs that it leaves to
  // the rollout and the host's rows (one layer with host buffers 371 -> 363 us, four at 236 of 2048 positions 812 -> 795).
  if (EPI != EPI_LMSTATS) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr bool kPairs = EPI == EPI_SWIGLU || EPI == EPI_QKV_ROPE;             // the epilogue pairs features
  const GemmArgs& g = p.g;
  const int cl = blockIdx.x >> 1;
  // The launch's record, or the row count if it has none (used behind the set-up, see below)
  int rec[24], n_live = 0;
  if (g.records) {
    const int4* from = reinterpret_cast<const int4*>(g.records + (size_t)cl * kWorkRecordBytes);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int4 x = __ldcg(from + q);
      rec[4 * q] = x.x; rec[4 * q + 1] = x.y; rec[4 * q + 2] = x.z; rec[4 * q + 3] = x.w;
    }
  } else {
    n_live = *reinterpret_cast<const volatile int32_t*>(g.n_rows);
  }
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* status = p.status ? p.status : g_tc_status;

  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = ((uint32_t)__cvta_generic_to_shared(smem_raw) + 1023u) & ~1023u;
  __shared__ __align__(8) uint64_t bars[2 * NST_MAX + 4];    // full[], empty[], acc_full[2], acc_empty[2]
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ __align__(8) float s_scale[MAX_TOK];
  __shared__ int s_pos[MAX_TOK], s_crow[MAX_TOK];
  __shared__ Part s_part[2];
  const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (NST_MAX + s); };
  auto acc_full = [&](int b) { return bar0 + 8u * (2 * NST_MAX + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (2 * NST_MAX + 2 + b); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST_MAX; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 2 * EPI_WARPS); }   // epilogue warps of both CTAs
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    prefetch_tensormap(&maps.w);
    if (EPI == EPI_SWIGLU) prefetch_tensormap(&maps.w2);
  }
  if (warp == 1) {
    tmem_alloc2((uint32_t)__cvta_generic_to_shared(&tmem_slot), 2 * MAX_TOK);
    tmem_relinquish2();
  }
  tc_fence_before();
  __syncwarp();
  cluster_arrive_all();                                      // (waited for below, behind arithmetic that needs neither)
  volatile int* abortp = &abort_flag;

  // The record or the row count is read, and the weight boxes of the first ring fill are requested, before the wait on the
  // preceding kernel: none is that kernel's output.  The count was written by the selection kernel at the start
  // of the step, and every kernel between it and a GEMM either waits for its own predecessor before it lets its
  // successor launch (the row kernels, attention) or is a GEMM behind such a kernel, so selection has completed
  // before any GEMM's CTA runs.  The records are the gather kernel's, behind it: the launch right behind that kernel, the first
  // layer's QKV projection, works its own out, and for all others a kernel that waits stands between.
  // Everything the predecessor may have written (activation rows, the residual, scratch)
  // is touched only behind each role's own griddepcontrol.wait.
  Tiling tl;
  WorkIter work;
  if (g.records) {
    unpack_record(rec, tl, work);
  } else {
    tl = Tiling(p.shape, n_live);
    work = WorkIter(tl, cl);
  }
  // Token boxes: each CTA brings in half of a tile's tokens.  The box is the smallest height that holds the widest
  // tile's half (rows beyond it are fetched and never multiplied); small boxes leave room for more stages.
  const int half_max = 8 * (tl.base + (tl.rem > 0 ? 1 : 0));
  int bi = 0;
  while (bi + 1 < N_BOXES && box_rows(bi) < half_max) ++bi;
  const uint32_t sub_bytes = W_BYTES + (uint32_t)box_rows(bi) * TK * 2, stage_bytes = KSUB * sub_bytes;
  const int nst = min(NST_MAX, (int)(RING_BYTES / stage_bytes));
  cluster_wait_all();                                        // both CTAs' barriers and accumulators exist
  tc_fence_after();
  const uint32_t tmem_acc = tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    // One lane per box: the weight boxes of the stage's first k-block and its token box, then those of the second.
    // The weights of the first ring fill are no output of the preceding kernel and do not wait for it; the activations that
    // go with them are another warp's work.
    constexpr int NBOX = (EPI == EPI_SWIGLU ? 2 : 1) + 1;     // SwiGLU: 64 gate rows and the 64 up rows of the same outputs
    const int u = lane / NBOX, bx = lane - u * NBOX;
    const bool is_tok = bx == NBOX - 1;
    const CUtensorMap* map = is_tok ? &maps.tok[bi] : (bx == 1 ? &maps.w2 : &maps.w);
    const uint32_t dst0 = smem_base + (uint32_t)u * sub_bytes + (is_tok ? (uint32_t)W_BYTES : (uint32_t)bx * (64u * TK * 2u));
    // Weights are read once per step (by clusters that run at the same time): they leave the L2 first, so that the stream
    // does not push out what the next kernels read, their instructions included.
    // (With many token tiles the readers of a block do not all run at once, and 28 layers at 3907 rows took 8 % longer.)
    const uint64_t policy = is_tok || tl.TT > 4 ? l2_policy_normal() : l2_policy_evict_first();
    bool ok = true;
    int nb, tile, k0, k1, kind;
    WorkIter w = work;
    uint32_t it = 0;                                          // stages issued so far
    int s = 0; uint32_t ph = 1;                               // ring position and the parity its empty barrier is waited for with
    while (ok && w.next(tl, nb, tile, k0, k1, kind)) {
      const int row = is_tok ? tl.tok0(tile) + (int)rank * (tl.width(tile) >> 1)
                             : (EPI == EPI_SWIGLU ? nb * 128 + (int)rank * 64 : nb * 256 + (int)rank * 128);
      for (int kt = k0; kt < k1; kt += KSUB, ++it) {
        const int nsub = min(KSUB, k1 - kt);
        if (it == (uint32_t)nst) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!__all_sync(0xffffffffu, mbar_wait(empty_bar(s), ph, abortp, status, 31))) { ok = false; break; }
        if (leader && lane == 0) mbar_expect_tx(full_bar(s), (uint32_t)nsub * 2u * sub_bytes);
        if (u < nsub && (!is_tok || it >= (uint32_t)nst)) tma_load_2d_pair(dst0 + s * stage_bytes, map, (kt + u) * TK, row, full_bar(s), policy);
        if (++s == nst) { s = 0; ph ^= 1; }
      }
    }
    if (EPI == EPI_LMSTATS) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (*abortp && leader && lane == 0) {
      for (uint32_t j = it > (uint32_t)nst ? it - nst : 0; j < it; ++j) {
        const long long t0 = clock64();
        while (!mbar_try_wait(full_bar(j % nst), (j / nst) & 1) && clock64() - t0 < kWaitCycles) {}
      }
    }
    __syncwarp();
  } else if (warp == TOKEN_WARP) {
    // ------------------------------------------------------------------ activations of the first ring fill (both CTAs)
    // One lane per k-block of a stage, as soon as the preceding kernel is done: behind the weights' warp, which is then
    // often still busy with its requests, the first MMA of a launch came 1.5 us later.
    const CUtensorMap* map = &maps.tok[bi];
    if (lane == 0) prefetch_tensormap(map);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // Launches take turns with two sets of meeting counters: this one clears the one before it, which is complete.  (Put back by the
    // last reader of each item, they cost the launch's end a barrier and an atomic's way to the L2 and back:
    // 32 layers at 80 rows 3870 -> 3820 us, 28 at 588 rows 9200 -> 9100.)
    if (g.sk_clear && blockIdx.x == 0)
      for (int i = lane; i < kPairCounters; i += 32) g.sk_clear[i] = 0;
    if (g.clock_probe && blockIdx.x == 0 && lane == 0) { g.clock_probe[0] = clock64(); g.clock_probe[1] = global_timer_ns(); }
    const uint32_t dst0 = smem_base + (uint32_t)lane * sub_bytes + (uint32_t)W_BYTES;
    const uint64_t policy = l2_policy_normal();
    int nb, tile, k0, k1, kind, s = 0;
    WorkIter w = work;
    while (s < nst && w.next(tl, nb, tile, k0, k1, kind)) {
      const int row = tl.tok0(tile) + (int)rank * (tl.width(tile) >> 1);
      for (int kt = k0; kt < k1 && s < nst; kt += KSUB, ++s)
        if (lane < min(KSUB, k1 - kt)) tma_load_2d_pair(dst0 + s * stage_bytes, map, (kt + lane) * TK, row, full_bar(s), policy);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (even CTA only)
    // The whole warp runs the loop and one lane's instructions take effect (see elect_one).  Under `if (lane == 0)` an MMA cost
    // about 58 clocks of issue, what the tensor cores need for 112 tokens: 32 layers at 80 rows 4095 -> 3985 us, two of d 512 at
    // 299 rows 133.7 -> 125.8, one of d 256 at 94 rows 59.2 -> 57.4.
    if (leader) {
      const uint32_t el = elect_one();
      uint32_t tcount = 0;
      bool ok = true;
      const uint64_t desc0 = smem_desc_sw128(smem_base);     // weights of stage 0, k-block 0
      const uint32_t sub_step = sub_bytes >> 4;
      int st = 0; uint32_t ph = 0;                           // ring position of the next stage
      WorkIter w = work;
      int nb, tile, k0, k1, kind;
      for (; ok && w.next(tl, nb, tile, k0, k1, kind); ++tcount) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(tl.width(tile) >> 3) << 17) | ((256u >> 4) << 24);
        const int nk = k1 - k0;
        const uint32_t buf = tcount & 1, use = tcount >> 1;
        if (!mbar_wait_warp(acc_empty(buf), (use & 1) ^ 1, abortp, status, 34)) { ok = false; break; }
        const uint32_t tacc = tmem_acc + buf * MAX_TOK;
        for (int j = 0; j < nk; j += KSUB) {
          const int nsub = min(KSUB, nk - j);
          if (!mbar_wait_warp(full_bar(st), ph, abortp, status, 32)) { ok = false; break; }
          tc_fence_after();
          const uint64_t wdesc = desc0 + (uint64_t)(st * (stage_bytes >> 4)), tdesc = wdesc + (W_BYTES >> 4);
#pragma unroll
          for (int u = 0; u < KSUB; ++u) {
            if (u < nsub) {
#pragma unroll
              for (int k = 0; k < TK / 16; ++k)               // +32 bytes per K=16 slice inside the swizzle atom
                umma2_bf16_e(el, tacc, wdesc + u * sub_step + 2 * k, tdesc + u * sub_step + 2 * k, idesc, (j | u | k) != 0);
            }
          }
          umma2_commit_pair_e(el, empty_bar(st), 3);          // both CTAs may refill this stage
          if (++st == nst) { st = 0; ph ^= 1; }
        }
        if (ok) umma2_commit_pair_e(el, acc_full(buf), 3);    // both CTAs' epilogues may read their rows
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int quarter = warp & 3;                             // TMEM lanes this warp may touch
    const int ehalf = (warp - 2) >> 2;                        // which half of a tile's token chunks it takes
    const int etid = (int)threadIdx.x - 64;
    const uint32_t stage_base = smem_base + RING_BYTES, stage = stage_base + (uint32_t)((warp - 2) * EPI_STAGE_BYTES);
    // paired features: the partner's lanes are 32 px lanes away, in another warp of the same half
    const int px = (EPI == EPI_QKV_ROPE && g.q_dh == 64) ? 1 : 2;
    const bool upper = kPairs && (quarter & px);
    const int lane_group = EPI == EPI_LMSTATS ? 0 : !kPairs ? quarter : (px == 2 ? quarter & 1 : quarter >> 1);        // warps that finish features together
    constexpr int NG = kPairs ? 2 : (EPI == EPI_LMSTATS ? 1 : 4);
    const uint32_t peer_stage = smem_base + RING_BYTES + (uint32_t)((((warp - 2) & 4) + (((quarter ^ px) + 2) & 3)) * EPI_STAGE_BYTES);
    auto first_feature = [&](int nb) {
      const int base = EPI == EPI_SWIGLU ? nb * 128 + (int)rank * 64 : nb * 256 + (int)rank * 128;
      return base + 32 * (kPairs ? (quarter & ~px) : quarter);
    };
    // Finishes tokens tk0 .. tk0 + 31.  Paired features: the lower warp keeps the first 16 tokens and hands over the
    // others, the upper warp the other way round; each thread swaps with the same lane of the other warp.
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(2 + ehalf * 2 + lane_group) : "memory"); };
    auto finish32 = [&](const EpiTile& e, float (&v)[32], int tk0, EpiPre<EPI>& pre, bool more) {
      if constexpr (!kPairs) {
        finish<EPI>(e, v, tk0, pre, more);
      } else {
        float x[32];
#pragma unroll
        for (int q = 0; q < 4; ++q) {                          // q = 2 h + j: four registers that stay, four that go
          const int a = 16 * (q >> 1) + 4 * (q & 1), b = a + 8;
          float4 give, have;
          give = upper ? make_float4(v[a], v[a + 1], v[a + 2], v[a + 3]) : make_float4(v[b], v[b + 1], v[b + 2], v[b + 3]);
          have = upper ? make_float4(v[b], v[b + 1], v[b + 2], v[b + 3]) : make_float4(v[a], v[a + 1], v[a + 2], v[a + 3]);
          sts128(stage + (uint32_t)(q * 512 + lane * 16), make_uint4(__float_as_uint(give.x), __float_as_uint(give.y), __float_as_uint(give.z), __float_as_uint(give.w)));
          x[4 * q] = have.x; x[4 * q + 1] = have.y; x[4 * q + 2] = have.z; x[4 * q + 3] = have.w;
        }
        pair_sync();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 t = lds128(peer_stage + (uint32_t)(q * 512 + lane * 16));
          const float4 o = make_float4(__uint_as_float(t.x), __uint_as_float(t.y), __uint_as_float(t.z), __uint_as_float(t.w));
          x[16 + 4 * q] = upper ? x[4 * q] : o.x; x[17 + 4 * q] = upper ? x[4 * q + 1] : o.y;
          x[18 + 4 * q] = upper ? x[4 * q + 2] : o.z; x[19 + 4 * q] = upper ? x[4 * q + 3] : o.w;
          if (upper) { x[4 * q] = o.x; x[4 * q + 1] = o.y; x[4 * q + 2] = o.z; x[4 * q + 3] = o.w; }
        }
        pair_sync();                                           // both have read: the buffers are free
        finish<EPI>(e, x, tk0 + (upper ? 16 : 0), pre, more);
      }
    };
    const int tk_mine = upper ? 16 : 0;                        // this warp's tokens of a chunk start here
    // What the epilogue needs per token of a tile (all epilogue warps together)
    int told_tile = -1;
    auto tell = [&](int tile, int n_end) {                    // rows from n_end on are not looked at
      const int t0 = tl.tok0(tile);
      if ((EPI != EPI_QKV_ROPE && !g.in_ssq) || tile == told_tile) return;
      told_tile = n_end > t0 ? tile : -1;
      asm volatile("bar.sync 1, 256;" ::: "memory");          // the previous tile's readers are done
      for (int i = etid; i < MAX_TOK; i += 32 * EPI_WARPS) {
        const int row = t0 + i;
        const bool live = row < n_end;
        if (g.in_ssq) {
          float s = 0.f;
          const int chunks = g.K >> 5;
          const float* sp = g.in_ssq + (size_t)row * chunks;
          if (live && (chunks & 3) == 0) {
#pragma unroll 8
            for (int t = 0; t < chunks; t += 4) {
              const float4 v = __ldcg(reinterpret_cast<const float4*>(sp + t));
              s += (v.x + v.y) + (v.z + v.w);
            }
          } else if (live) {
            for (int t = 0; t < chunks; ++t) s += __ldcg(sp + t);
          }
          s_scale[i] = rsqrtf(s / (float)g.K + g.in_eps);
        }
        if (EPI == EPI_QKV_ROPE) {
          const int pos = live ? g.q_sel_idx[row] : 0;
          s_pos[i] = pos;
          s_crow[i] = live ? g.q_row_seq[row] * g.q_cache_seq + pos : 0;
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    };
    int pending = work.parts();
    const bool keep = !work.has_whole();                      // nothing follows the parts: their sums can wait in TMEM
    const int n_acc = pending + (keep ? 0 : div24(work.unit_end - 1 - work.unit, work.G) + 1);      // accumulators of this cluster
    // this cluster's parts, in the order of its accumulators; worked out while the main loop runs
    const int q_me = work.unit, member = work.j, n_part = pending;
    if (etid < n_part) {
      const int unit = (work.s_tail1 > work.s_tail0 ? work.u_tail : work.u_head) - tl.F * tl.G + etid;      // among the shared ones
      Part t;
      const int u = tl.F * tl.G + unit;
      if (tl.GS == 1) tl.item(u, t.nb, t.tile); else { t.nb = u; t.tile = member; }
      t.g0 = tl.group_of(unit * tl.KS);
      t.parts = tl.group_of((unit + 1) * tl.KS - 1) - t.g0 + 1;
      t.mine = q_me - t.g0;
      const int cells = ((min(tl.n - tl.tok0(t.tile), tl.width(t.tile)) + 15) >> 4) * NG;      // shared evenly
      t.a0 = div24(cells * t.mine, t.parts); t.a1 = div24(cells * (t.mine + 1), t.parts);
      s_part[etid] = t;
    }
    if (n_part > 0) asm volatile("bar.sync 1, 256;" ::: "memory");
    const float4* parked = reinterpret_cast<const float4*>(g.sk_partials) + (size_t)rank * SLOT_F4;
    auto slot_of = [&](int cluster, bool head) { return (size_t)((cluster * 2 + (head ? 1 : 0)) * 2) * SLOT_F4; };
    // The warp reads TMEM no more.  The CTAs of the pair part here, ahead of the last items' arithmetic and stores, which then run
    // beside the wait for the peer and the release of TMEM (before, 0.7 us of a launch behind them: 32 layers at 80 rows 3931 -> 3894
    // us, two of d 512 at 299 rows 127.4 -> 124.4, and that although the LM head and the residual form spill two to four registers
    // more for it).  Relaxed: what is stored need not be seen by the peer, and a release would wait for it.
    bool left_tmem = false;
    auto leave_tmem = [&]() {
      tc_fence_before();
      __syncwarp();
      if (!left_tmem) cluster_arrive_relaxed();
      left_tmem = true;
    };
    // The loop's first round is a rehearsal without live rows, before the wait on the preceding kernel: it reads and writes
    // nothing of the step's and brings the epilogue's instructions in.  A step streams its weights through the L2 between
    // two launches of the same kernel; met for the first time behind the last MMA, the code cost about 3 us of a launch,
    // and behind that wait up to 5 us of one with few stages.
    WorkIter w = work;
    int nb = 0, tile = 0, k0 = 0, k1 = 0, kind = WARM;
    { WorkIter first = work; int kd; if (!first.next(tl, nb, tile, k0, k1, kd)) w.unit_end = 0; }
    for (int round = -1;; ++round) {
      // the residual, the scratch and the outputs belong to the step's chain (and every CTA waits, with work or without:
      // a launch must not be over before its predecessor)
      if (round == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
      if (round >= 0 && !w.next(tl, nb, tile, k0, k1, kind)) break;
      const uint32_t buf = round & 1, use = (uint32_t)round >> 1;
      const int t0 = tl.tok0(tile), n_end = min(tl.n, t0 + tl.width(tile)), live_tok = n_end - t0;
      tell(tile, kind == WARM ? t0 : n_end);
      const int chunks = (live_tok + 31) >> 5, c_mid = (chunks + 1) >> 1;
      const int c0 = ehalf ? c_mid : 0, c1 = ehalf ? chunks : c_mid;
      // what this warp finishes: units [ua, ub) of 16 tokens
      int ua = 2 * c0, ub = 2 * c1, ejob_nb = nb, ejob_t0 = t0, ejob_n = n_end;
      if (kind == WARM) { ua = 0; ub = 2; ejob_n = t0; }
      EpiPre<EPI> pre;
      auto job = [&]() { return EpiTile{g, ejob_t0, ejob_n, lane, first_feature(ejob_nb), stage, stage_base, g.in_ssq ? s_scale : nullptr, s_pos, s_crow,
                                         stage_base + (uint32_t)(ehalf * 4 * EPI_STAGE_BYTES), quarter, ejob_nb * 2 + (int)rank}; };
      if ((kind == FULL || kind == WARM) && ua < ub) pre.load(job(), ua * 16 + tk_mine);
      const uint32_t tbase = tmem_acc + buf * MAX_TOK + ((uint32_t)(quarter * 32) << 16);
      auto load_acc = [&](uint32_t at, float (&v)[32]) {      // 32 columns of this warp's 32 lanes
        uint32_t r[32];
        tmem_ld_16x32(at, r);
        tmem_ld_16x32(at + (16u << 16), r + 16);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
      };
      // This warp has read its part of the accumulator.  (Nobody waits for the last two to be read.)
      auto release_acc = [&]() {
        tc_fence_before();
        __syncwarp();
        if (round + 2 < n_acc) { if (lane == 0) mbar_arrive_even_cta(acc_empty(buf)); }
        else if (round + 1 == n_acc) leave_tmem();
      };
      int jobs = 1;
      if (kind != WARM) {
        // a wait that gave up ends the loop for the whole warp (the tcgen05.ld below is warp-collective) and, since the
        // epilogue warps meet at named barriers, for all of them together
        const bool got = mbar_wait(acc_full(buf), use & 1, abortp, status, 33);
        if (meet_or_leave<1, 256>(!got)) break;
        tc_fence_after();
        if (kind != FULL) {
          // ---- a part of a split item: park what the other contributors will finish
          const Part me = s_part[round];
          const int cells = ((live_tok + 15) >> 4) * NG;
          float4* slot = reinterpret_cast<float4*>(g.sk_partials) + (size_t)rank * SLOT_F4 + slot_of(cl, kind == HEAD);
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            float v[32];
            load_acc(tbase + c * 32, v);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int u = 2 * c + h, cell = u * NG + lane_group;
              if (cell < cells && !(keep && cell >= me.a0 && cell < me.a1)) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const int i = 16 * (q >> 1) + 8 * h + 4 * (q & 1);
                  __stcg(slot + (size_t)((u * 4 + quarter) * 4 + q) * 32 + lane, make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]));
                }
              }
            }
          }
          if (!keep) release_acc();
          asm volatile("bar.sync 1, 256;" ::: "memory");
          if (etid == 0)                                       // (the release covers what the barrier has ordered before it)
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(g.sk_counters + (me.g0 * tl.GS + member) * 2 + (int)rank) : "memory");      // counted at the cluster that holds the item's start
          if (--pending > 0) continue;
          jobs = n_part;                                       // every part of this cluster is parked: finish its cells of each
        }
      }
#pragma unroll 1
      for (int r = 0; r < jobs; ++r) {
        int parts = 0, mine = 0, g0 = 0;
        if (kind == TAIL || kind == HEAD) {
          const Part me = s_part[r];
          parts = me.parts; mine = me.mine; g0 = me.g0;
          ejob_t0 = tl.tok0(me.tile); ejob_nb = me.nb;
          // units u with a0 <= NG u + lane_group < a1, half of them for each of the two warps
          if (NG == 4) { ua = (me.a0 - lane_group + 3) >> 2; ub = (me.a1 - lane_group + 3) >> 2; }
          else if (NG == 2) { ua = (me.a0 - lane_group + 1) >> 1; ub = (me.a1 - lane_group + 1) >> 1; }
          else { ua = me.a0; ub = me.a1; }
          const int um = (ua + ub + 1) >> 1;
          if (ehalf) ua = um; else ub = um;
          ejob_n = min(min(tl.n, ejob_t0 + tl.width(me.tile)), ejob_t0 + ub * 16);
          tell(me.tile, min(tl.n, ejob_t0 + tl.width(me.tile)));
          if (EPI != EPI_QKV_ROPE && ua < ub) pre.load(job(), ua * 16 + tk_mine);
          if (etid == 0) {
            const int32_t* cnt = g.sk_counters + (g0 * tl.GS + member) * 2 + (int)rank;
            const long long tw = clock64();
            for (;;) {
              int32_t come;
              asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(come) : "l"(cnt) : "memory");
              if (come >= parts || *abortp) break;
              if (clock64() - tw > kWaitCycles) {
                *abortp = 1;
                if (atomicCAS(status, 0, D2C_ETIMEOUT) == 0) status[1] = 35;
                break;
              }
            }
          }
          if (meet_or_leave<1, 256>(*abortp != 0)) goto leave;
        }
        const EpiTile e = job();
#pragma unroll 1
        for (int u2 = ua; u2 < ub; u2 += 2) {
          float v[32];
          bool ahead = u2 + 2 < ub;                            // ask for the next chunk's operands while this one is finished
          if (kind == FULL) {
            load_acc(tbase + u2 * 16, v);
            if (!ahead) release_acc();
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0.f;
            const bool two = u2 + 1 < ub;
            const float4* sp = parked + (size_t)((u2 * 4 + quarter) * 4) * 32 + lane;
#pragma unroll 1
            for (int p0 = 0; p0 < parts; p0 += 2) {            // in part order, two parts' loads in flight
              float4 x[2][8];
#pragma unroll
              for (int d = 0; d < 2; ++d) {                    // the first part is its cluster's HEAD, the others are TAILs
                const int pt = p0 + d;
                const bool rd = pt < parts && !(keep && pt == mine);
                const float4* pp = sp + slot_of((g0 + pt) * tl.GS + member, pt == 0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  x[d][q] = rd ? __ldcg(pp + q * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
                  x[d][4 + q] = rd && two ? __ldcg(pp + 512 + q * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
              }
#pragma unroll
              for (int d = 0; d < 2; ++d) {
                if (keep && p0 + d == mine) {                  // (part r of a cluster is its r-th accumulator)
                  float y[32];
                  load_acc(tmem_acc + (uint32_t)r * MAX_TOK + ((uint32_t)(quarter * 32) << 16) + u2 * 16, y);
#pragma unroll
                  for (int i = 0; i < 32; ++i) v[i] += y[i];
                } else {
#pragma unroll
                  for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                      const int i = 16 * (q >> 1) + 8 * h + 4 * (q & 1);
                      const float4 y = x[d][4 * h + q];
                      v[i] += y.x; v[i + 1] += y.y; v[i + 2] += y.z; v[i + 3] += y.w;
                    }
                }
              }
            }
            if (EPI == EPI_QKV_ROPE) { pre.load(e, u2 * 16 + tk_mine); ahead = false; }       // (they would not fit beside the parts)
            if (keep && r + 1 == jobs && u2 + 2 >= ub) leave_tmem();
          }
          finish32(e, v, u2 * 16, pre, ahead);
        }
        if (kind == FULL && ua >= ub) {
          release_acc();
        }
      }
    }
  leave:
    leave_tmem();
    if (g.clock_probe && blockIdx.x == 0 && etid == 0) { g.clock_probe[2] = clock64(); g.clock_probe[3] = global_timer_ns(); }
    return;
  }
  // ------------------------------------------------------------------ teardown (loads, MMAs)
  tc_fence_before();
  __syncwarp();
  cluster_arrive_relaxed();
  if (warp == 1) {
    cluster_wait_all();                                      // nobody reads TMEM any more, nor signals a CTA of the pair
    tc_fence_after();
    tmem_dealloc2(tmem_acc, 2 * MAX_TOK);
  }
}

template <int EPI>
int launch_one(const GemmArgs& g, int* status, cudaStream_t st) {
  const int smem = RING_BYTES + 1024 + EPI_WARPS * EPI_STAGE_BYTES;    // stage ring, alignment slack, epilogue buffers
  static PerDevice attr_set;
  if (attr_set.first()) {
    D2C_CUDA_OK(cudaFuncSetAttribute(gemm_tc2_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  }
  Tc2Maps fresh, *m = &fresh;
  static_assert(sizeof(Tc2Maps) <= sizeof(MapCache::maps), "the cache holds one launch's maps");
  bool made = false;
  if (g.cache) {
    m = reinterpret_cast<Tc2Maps*>(g.cache->maps);
    made = g.cache->same(g.A, g.W, g.W2, g.max_rows, g.N, g.K, g.lda, EPI, 2);
  }
  if (!made) {
    const uint32_t wbox = EPI == EPI_SWIGLU ? 64 : 128;
    int rc = make_bf16_map(&m->w, g.W, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)g.K, wbox);
    if (rc == D2C_OK) rc = make_bf16_map(&m->w2, EPI == EPI_SWIGLU ? g.W2 : g.W, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)g.K, wbox);
    for (int i = 0; i < N_BOXES && rc == D2C_OK; ++i)
      rc = make_bf16_map(&m->tok[i], g.A, (uint64_t)g.max_rows, (uint64_t)g.K, (uint64_t)g.lda, (uint32_t)box_rows(i));
    if (rc != D2C_OK) { if (g.cache) g.cache->forget(); return rc; }
  }
  Tc2Params p{g, gemm_tc2_shape(g, (GemmEpilogue)EPI), status};
  const int ctas = 2 * p.shape.clusters;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(TC_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  D2C_CUDA_OK(cudaLaunchKernelEx(&cfg, gemm_tc2_kernel<EPI>, *m, p));
  count_launch(1);
  return D2C_OK;
}
}  // namespace

// Shapes the pair kernel takes; everything else goes to the one-SM kernel.
bool gemm_tc2_supported(const GemmArgs& g) {
  return g.max_rows >= kPairRows && g.N >= 256 && g.K % TK == 0 && (g.lda & 7) == 0 && (g.N & 1) == 0 && (g.ldc & 1) == 0 &&
         (reinterpret_cast<uintptr_t>(g.A) & 15) == 0 && (reinterpret_cast<uintptr_t>(g.W) & 15) == 0;
}

int launch_gemm_tc2(const GemmArgs& g, GemmEpilogue epi, cudaStream_t st, int* status) {
  switch (epi) {
    case EPI_STORE: return launch_one<EPI_STORE>(g, status, st);
    case EPI_RESIDUAL: return launch_one<EPI_RESIDUAL>(g, status, st);
    case EPI_SWIGLU: return launch_one<EPI_SWIGLU>(g, status, st);
    case EPI_QKV_ROPE: return launch_one<EPI_QKV_ROPE>(g, status, st);
    case EPI_LMSTATS: return launch_one<EPI_LMSTATS>(g, status, st);
  }
  return D2C_EINVAL;
}

}  // namespace d2c

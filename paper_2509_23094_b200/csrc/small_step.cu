// The whole step of a small model in one launch.
//
// A step of a model of a few layers of d 256 to 512 is a chain of 8 to 26 dependent kernels of 1 to 3 us of work each; launched one
// by one they cost 4 to 9 us apiece, and the host needs as long to enqueue them.  Here clusters of 16 CTAs stay from the selection to
// the rollout.  A cluster takes an equal share of the selected rows, in tiles of 16 of one sequence, and does everything that is local
// to rows (norms, projections, its queries' attention, FFN, LM head) by itself: each of its CTAs a sixteenth of the output columns,
// with a cluster barrier (0.35 us) between products.  Only what crosses rows meets the whole grid (1.3 us): the selected set, each
// layer's K/V, and each layer of the rollout.
//
// What bounds it is latency: the L2's (0.4 us a dependent load), the barriers' and that of fetching instructions that run once or a few
// times.  So products are shaped for few dependent steps and not for the rate of the matrix unit: a warp holds a piece of the weights, 16
// columns x up to 256 of K, in registers, requested
// before the barrier that its activations wait for, and multiplies it with every tile of rows (mma.sync; tcgen05 would add the trips
// into shared memory and out of TMEM, and tiles of 128 rows where a cluster has 16 to 64).  Keys and values come straight from
// the L2 into fragments.  Both are read 16 bytes a lane: the order of K inside a product is free, so lane q of a group of four takes
// eight neighbouring elements of a row, and two MMAs' fragments are the two halves of what it has.
//
// Measured (us a step, this launch / the separate kernels; one layer of d 256, 94 rows of 128 positions: 41 / 52): 256 threads a CTA
// 41, 512 52 (barriers; half of the instructions are per warp); rows by bulk copies 2 a product more than by cp.async; a normed row
// pushed into the other CTAs' shared memory 44; keys of a unit shared by several CTAs and merged: 0 to 9 more up to 2100 positions, 2 to 8 %
// less at 4096; heads of 128, which need twice the registers for V and Q: 5 to 15 % ahead of the separate kernels up to 130 rows only, so left to them.
//
// Compiled without fast math, as the selection decides indices from fp32 products.
#include "select_seq.cuh"
#include "sm100_ptx.cuh"

namespace d2c {
namespace {

constexpr int CL = kSmallCluster;                 // CTAs of a cluster
constexpr int NT = 256, NW = NT / 32;             // threads and warps of a CTA
constexpr int P = 8;                              // row tiles of a pass at most
constexpr int CB = 8;                             // 32-wide blocks of K that a warp holds of its weights
constexpr int DH = 64;                            // head dimension
constexpr int MAXT = kSmallMaxTiles;              // row tiles of a cluster at most
constexpr int MAXB = kSmallMaxBatch;
constexpr int kPosMask = (1 << kPosBits) - 1;
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
constexpr float kNoKey = -3e38f;                  // maximum before the first score: finite, as scores may be -inf
constexpr int RT = NW * 256;                      // floats of a tile's partial sums
constexpr int kGain = 2048, kProb = NW * 512 * 4, kPassBytes = kSmallSmem - kGain - kProb;      // bytes: a row of gains; the probabilities' sums; a pass's sums and rows

__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 32 of K: x and y hold rows g and g + 8 of A, b a row of B, eight elements a lane each.
__device__ __forceinline__ void mma_k32(float (&c)[4], const uint4& x, const uint4& y, const uint4& b) {
  mma16816(c, x.x, y.x, x.y, y.y, b.x, b.y);
  mma16816(c, x.z, y.z, x.w, y.w, b.z, b.w);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float2 unpack2(uint32_t u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); }
__device__ __forceinline__ uint4 ldcg16(const bf16* p) { return __ldcg(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ uint4 ldw16(const bf16* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ void copy16(void* to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---- barriers ----------------------------------------------------------------------------------
// (.aligned: all threads of a warp together.  Most of them come out of loops whose trip counts differ inside a warp.)
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// All CTAs of the grid, which a cooperative launch keeps on the GPU together.  The wait is bounded: behind one that gave up the CTA
// goes on without waiting, so all barriers are still reached, and the step's status tells.  Behind the first, which all others' indices
// come from, it has no rows and takes no index from memory; what later ones let through are values.
struct Grid {
  uint32_t* count; int* status; uint32_t due; bool dead;             // dead: in thread 0
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    due += gridDim.x;
  }
  __device__ __forceinline__ void wait(int site) {
    if (threadIdx.x == 0 && !dead) {
      const long long t0 = clock64();
#pragma unroll 1
      for (;;) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
        if ((int)(v - due) >= 0) break;
        if (clock64() - t0 > kWaitCycles) {
          dead = true;
          if (atomicCAS(status, 0, D2C_ETIMEOUT) == 0) status[1] = site;
          break;
        }
      }
    }
    __syncthreads();
  }
};

// a / b for small a >= 0, b > 0 (an integer division is a chain of some forty dependent instructions)
__device__ __forceinline__ int quot(int a, int b) {
  const int q = __float2int_rz(__fdividef((float)a, (float)b)), r = a - q * b;
  return q + (r >= b ? 1 : 0) - (r < 0 ? 1 : 0);
}

// The products of a step: four of each layer, and the LM head.
enum Step { S_QKV = 0, S_O = 1, S_GATEUP = 2, S_DOWN = 3, S_LM = 4 };

// The cluster's size is the kernel's own, not an attribute of its launch: a tool that launches the kernel in its own way (ncu) kept the
// cooperative attribute and left that one out, and clusters of one CTA meet every barrier and write a sixteenth of the results.
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT, 1) small_step_kernel(const __grid_constant__ SmallArgs a) {
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ int s_off[MAXB + 1], s_lmoff[MAXB + 1], s_toff[MAXB + 1], s_ct[kSmallMaxClusters + 1];
  __shared__ int4 s_tile[MAXT];                    // first row, rows, sequence, first row of the sequence's cache
  __shared__ int s_pos[MAXT * 16];                 // position | (rank among the masked rows + 1) << kPosBits
  __shared__ int s_lm[MAXT * 16];                  // rows that go through the LM head: slot (tile * 16 + row)
  __shared__ float s_u[MAXT * 16];
  __shared__ float s_f[NW * 16];
  __shared__ float s_mx[P * 16], s_sum[P * 16];
  __shared__ int s_arg[P * 16];
  __shared__ int s_lmlo, s_lmn;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, q = lane & 3;
  const int rank = (int)cluster_ctarank(), cidx = blockIdx.x / CL, ncl = gridDim.x / CL;
  const int B = a.sel.batch, L = a.sel.seq_len, d = a.d, hq = a.hq, n_layers = a.n_layers;
  // (in another cluster nothing is begun: all CTAs leave, and the status tells)
  if (cluster_size() != CL) {
    if (blockIdx.x == 0 && tid == 0 && atomicCAS(a.status, 0, D2C_ECUDA) == 0) { a.status[1] = 63; a.status[2] = (int)cluster_size(); }
    return;
  }
  constexpr int UH = DH / 16;                      // units of a head: eight columns of its low half, eight of its high half
  const int d_o = hq * DH, kv_ld = a.hkv * DH;
  unsigned char* s_gain = dyn;
  float* red = reinterpret_cast<float*>(dyn + kGain);          // [pt][NW][16][16]: partial sums of the parts of K; scratch between products
  float* s_p = reinterpret_cast<float*>(dyn + kGain + kPassBytes);      // [warp][16][32]
  Grid grid{a.sync, a.status, 0u, false};
  if (tid == 0) { s_lmlo = 0x7fffffff; s_lmn = 0; }

  // ---- selection: sequence b by CTA b / clusters of cluster b % clusters ------------------------------
  if (rank * ncl + cidx < B) {
    select_sequence<true, NT>(a.sel, rank * ncl + cidx, dyn);
  } else {
    // (the arguments' first use in an SM is a miss in the constant cache: taken while there is nothing to do)
    uint32_t x = 0;
#pragma unroll 1
    for (int i = 16 * lane; i < (int)(sizeof(SmallArgs) / 4); i += 512) x ^= reinterpret_cast<const uint32_t*>(&a)[i];
    asm volatile("" ::"r"(x));
  }
  grid.arrive();

  // A CTA's share of a product: units of 16 weight rows (lo: eight, hi: eight that belong to them), to each warp one unit of a group and
  // a part of K (a power of two of them, as many as there are warps for), of which it holds up to CB blocks of 32.
  int K = d, u0 = 0, units = 0, lks = 0, per = NW, ul = 0, b0 = 0, nb = 0;      // first unit and units; log2 of the parts; units of a group; this warp's unit and blocks
  uint4 lo[CB], hi[CB];
  const bf16 *plo = nullptr, *phi = nullptr;
  const bf16 *w_lo = nullptr, *w_hi = nullptr;                 // row g8 of unit 0, in this lane's 16 bytes of the warp's first block
  auto load_blocks = [&](int b) {
#pragma unroll
    for (int i = 0; i < CB; ++i) {
      if (b + i < nb) { lo[i] = ldw16(plo + 32 * (b + i)); hi[i] = ldw16(phi + 32 * (b + i)); }
      else lo[i] = hi[i] = make_uint4(0, 0, 0, 0);
    }
  };
  auto request = [&](int step, int g) {                        // the weights of unit g + ul
    const int U = u0 + g + ul;
    int row;                                                   // of the unit's first weight row
    if (step == S_QKV) { const int h = U / UH; row = h * DH + 8 * (U - h * UH); }
    else row = step == S_GATEUP ? 8 * U : 16 * U;
    plo = w_lo + row * K; phi = w_hi + row * K;
    if (step == S_LM) {
      const int last = a.vocab - 1;
      plo = w_lo + (min(row + g8, last) - g8) * K; phi = w_lo + (min(row + 8 + g8, last) - g8) * K;
    }
    if (g + ul >= units) return;
    load_blocks(0);
  };
  auto begin = [&](int step, int l) {
    const SmallLayer& y = a.layer[l];
    const bf16 *w = y.wqkv, *gain = y.g_attn;
    int n = (hq + 2 * a.hkv) * UH, apart = DH / 2;             // units; rows between a unit's halves
    K = d;
    if (step == S_O) { w = y.wo; n = d >> 4; K = d_o; apart = 8; gain = nullptr; }
    if (step == S_GATEUP) { w = y.w_gate; n = a.ffn >> 3; gain = y.g_ffn; }
    if (step == S_DOWN) { w = y.w_down; n = d >> 4; K = a.ffn; apart = 8; gain = nullptr; }
    if (step == S_LM) { w = a.w_lm; n = (a.vocab + 15) >> 4; gain = a.g_final; }
    const int kb = K >> 5;
    u0 = rank * n / CL; units = (rank + 1) * n / CL - u0;
    lks = min(units > 4 ? 0 : 3 - (units > 1 ? 32 - __clz(units - 1) : 0), 31 - __clz(kb));
    per = NW >> lks; ul = warp >> lks;
    const int split = warp & ((1 << lks) - 1);
    b0 = split * kb >> lks; nb = ((split + 1) * kb >> lks) - b0;
    const int at = g8 * K + 32 * b0 + 8 * q;
    w_lo = w + at; w_hi = step == S_GATEUP ? y.w_up + at : w_lo + apart * K;
    request(step, 0);
    if (gain && tid < K >> 3) copy16(s_gain + 16 * tid, gain + 8 * tid);
  };
  begin(S_QKV, 0);
  grid.wait(60);

  // ---- the rows of this cluster ----------------------------------------------------------------------
  if (warp == 0) {
    int n = 0, m = 0;
    const bool lost = __shfl_sync(0xffffffffu, grid.dead, 0);      // nothing is known of the selection
    if (lane < B && !lost) { n = min(max(__ldcg(a.sel.n_b + lane), 0), L); m = min(max(__ldcg(a.sel.nm_b + lane), 0), n); }
    int t = (n + 15) >> 4, sn = n, sm = m, st = t;
#pragma unroll 1
    for (int o = 1; o < B; o <<= 1) {
      const int un = __shfl_up_sync(0xffffffffu, sn, o), um = __shfl_up_sync(0xffffffffu, sm, o), ut = __shfl_up_sync(0xffffffffu, st, o);
      if (lane >= o) { sn += un; sm += um; st += ut; }
    }
    if (lane < B) { s_off[lane + 1] = sn; s_lmoff[lane + 1] = sm; s_toff[lane + 1] = st; }
    if (lane == 0) s_off[0] = s_lmoff[0] = s_toff[0] = 0;
    const int total = __shfl_sync(0xffffffffu, st, B - 1);
    if (lane <= ncl) s_ct[lane] = quot(lane * total, ncl);     // first tile of each cluster
    if (lane == B - 1 && blockIdx.x == 0 && a.n_word)
      // (64 bits at once: of a vector store the host may see one half before the other)
      asm volatile("st.relaxed.sys.global.u64 [%0], %1;" ::"l"(a.n_word), "l"((unsigned long long)(uint32_t)a.n_tag << 32 | (uint32_t)sn) : "memory");
  }
  __syncthreads();
  const int t0 = s_ct[cidx], mt = min(s_ct[cidx + 1] - t0, MAXT);
#pragma unroll 1
  for (int i = tid; i < mt * 16; i += NT) {
    const int t = t0 + (i >> 4), r = i & 15;
    int b = 0;
#pragma unroll 1
    while (t >= s_toff[b + 1]) ++b;
    const int rb = 16 * (t - s_toff[b]), n = s_off[b + 1] - s_off[b];
    if (r == 0) s_tile[i >> 4] = make_int4(s_off[b] + rb, min(16, n - rb), b, b * a.cache_seq);
    int v = 0;
    if (rb + r < n) {
      v = __ldcg(a.sel.rank_s + b * L + rb + r);
      const int pos = min(v & kPosMask, L - 1), rl = min(max((v >> kPosBits) - 1, -1), s_lmoff[b + 1] - s_lmoff[b] - 1);
      v = pos | ((rl + 1) << kPosBits);
    }
    s_pos[i] = v; s_u[i] = 1.f;
  }
  __syncthreads();
  // What only later phases and the caller need of the selection, behind the first projections.
  auto publish_rows = [&]() {
    const int n_total = s_off[B];
    if (blockIdx.x == 0 && tid <= B) {
      a.sel.row_off[tid] = s_off[tid]; a.sel.lm_off[tid] = s_lmoff[tid];
      if (a.copies.dst[1]) a.copies.dst[1][tid] = s_off[tid];
    }
    if (blockIdx.x == gridDim.x - 1) {
#pragma unroll 1
      for (int i = tid; i < a.n_clear; i += NT) a.clear[i] = 0;
      if (a.copies.dst[0])                                     // (whatever lies behind the rows, as the copy of the whole array has it)
#pragma unroll 1
        for (int i = n_total + tid; i < a.copies.n[0]; i += NT) a.copies.dst[0][i] = a.sel.sel_idx[i];
    }
#pragma unroll 1
    for (int i = tid; i < mt * 16; i += NT) {
      const int4 t = s_tile[i >> 4];
      if ((i & 15) >= t.y) continue;
      const int rl = (s_pos[i] >> kPosBits) - 1, pos = s_pos[i] & kPosMask, lm = rl >= 0 ? s_lmoff[t.z] + rl : -1, row = t.x + (i & 15);
      if (lm >= 0) { atomicMin(&s_lmlo, lm); atomicAdd(&s_lmn, 1); }
      if (rank == (i & 15)) {                                  // (a row of each tile to a CTA)
        a.sel.sel_idx[row] = pos; a.sel.row_seq[row] = t.z; a.sel.slot_of_pos[t.z * L + pos] = row;
        if (lm >= 0) a.sel.lm_rows[lm] = row;
        if (a.copies.dst[0]) a.copies.dst[0][row] = pos;
      }
    }
    __syncthreads();
    const int n = s_lmn;
#pragma unroll 1
    for (int i = tid; i < mt * 16; i += NT) {
      const int rl = (s_pos[i] >> kPosBits) - 1, at = s_lmoff[s_tile[i >> 4].z] + rl - s_lmlo;
      if (rl >= 0 && (i & 15) < s_tile[i >> 4].y && at >= 0 && at < n) s_lm[at] = i;
    }
  };

  // Attention by units, a tile's rows in one head each.
  const int nu = mt * hq, ua = rank * nu / CL, ub = (rank + 1) * nu / CL;
  const float sc = kLog2e * rsqrtf((float)DH);
  const int group = quot(hq, a.hkv);
  // And the probabilities: hw heads' warps share a tile's rows x 32 keys, cg such pieces to a CTA at a time
  const int hw = min(hq, NW), wg = quot(warp, hw), wh = warp - wg * hw, cg = quot(NW, hw), ck = (L + 31) >> 5;

  // Rollout: u_i * Abar[i][j] summed over this cluster's rows of each sequence, this CTA's columns.
  auto rollout_sums = [&](int l) {
    const int step = (L + CL - 1) / CL, j0 = min(L, rank * step), cols = min(L, j0 + step) - j0;
    const int lcw = cols > 16 ? 5 : cols > 8 ? 4 : 3, cw = 1 << lcw, rs = lane >> lcw, dr = NW << (5 - lcw), rg = (warp << (5 - lcw)) + rs;
    const float* abar = a.abar + (size_t)l * a.abar_layer;
#pragma unroll 1
    for (int ta = 0; ta < mt;) {
      const int4 first = s_tile[ta];
      int tb = ta, nr = 0;
#pragma unroll 1
      while (tb < mt && s_tile[tb].z == first.z) nr += s_tile[tb++].y;
#pragma unroll 1
      for (int c0 = 0; c0 < cols; c0 += cw) {
        const int j = c0 + (lane & (cw - 1));
        float acc = 0.f;
        if (j < cols) {
          const float* p = abar + (first.x + rg) * L + j0 + j;
          const float* uu = s_u + 16 * ta;
#pragma unroll 4
          for (int i = rg; i < nr; i += dr, p += dr * L) acc += uu[i] * __ldcg(p);
        }
#pragma unroll 1
        for (int o = cw; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (rs == 0) red[warp * cw + lane] = acc;
        __syncthreads();
        if (tid < cw && c0 + tid < cols) {
          float s = 0.f;
#pragma unroll
          for (int x = 0; x < NW; ++x) s += red[x * cw + tid];
          a.rp[((l * ncl + cidx) * B + first.z) * L + j0 + c0 + tid] = s;
        }
        __syncthreads();
      }
      ta = tb;
    }
  };
  auto sum_over_clusters = [&](int l, int b, int j) {          // of those with rows of sequence b
    float s = 0.f;
    const float* p = a.rp + (l * ncl * B + b) * L + j;
    const int lo_t = s_toff[b], hi_t = s_toff[b + 1];
#pragma unroll 1
    for (int c0 = 0; c0 < ncl; c0 += 4) {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = c0 + k;
        v[k] = c < ncl && max(s_ct[c], lo_t) < min(s_ct[min(c, ncl - 1) + 1], hi_t) ? __ldcg(p + c * B * L) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) s += v[k];
    }
    return s;
  };

  // ---- head-averaged probabilities, while the output projection's rows are on their way: 16 rows x 32 keys of one head to a warp ----
  auto probabilities = [&](int l, const bf16* kc) {
    const int pairs = mt * ck;
    const float invh = 1.f / (float)hq;
    float* abar = a.abar + (size_t)l * a.abar_layer;
#pragma unroll 1
    for (int i0 = rank * cg; i0 < pairs; i0 += CL * cg) {
      const int pi = i0 + wg;
      if (wg < cg && pi < pairs) {
        const int t = quot(pi, ck), k0 = 32 * (pi - t * ck);
        const int4 tile = s_tile[t];
        float p[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j][0] = p[j][1] = p[j][2] = p[j][3] = 0.f;
#pragma unroll 1
        for (int h = wh; h < hq; h += hw) {
          const int r0 = min(g8, tile.y - 1), r1 = min(g8 + 8, tile.y - 1);
          const bf16* qp = a.q + tile.x * d_o + h * DH + 8 * q;
          const bf16* kb = kc + tile.w * kv_ld + quot(h, group) * DH + 8 * q;
          uint4 qx[DH / 32], qy[DH / 32];
#pragma unroll
          for (int i = 0; i < DH / 32; ++i) { qx[i] = ldcg16(qp + r0 * d_o + 32 * i); qy[i] = ldcg16(qp + r1 * d_o + 32 * i); }
          const float e0 = kLog2e * __ldcg(a.lse + (tile.x + r0) * hq + h), e1 = kLog2e * __ldcg(a.lse + (tile.x + r1) * hq + h);
          uint4 kf[4][DH / 32];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const bf16* kp = kb + min(k0 + 8 * j + g8, L - 1) * kv_ld;
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) kf[j][i] = ldcg16(kp + 32 * i);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) mma_k32(s, qx[i], qy[i], kf[j][i]);
            p[j][0] += ex2(s[0] * sc - e0); p[j][1] += ex2(s[1] * sc - e0); p[j][2] += ex2(s[2] * sc - e1); p[j][3] += ex2(s[3] * sc - e1);
          }
        }
        float* to = s_p + (warp * 16 + g8) * 32 + 2 * q;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          *reinterpret_cast<float2*>(to + 8 * j) = make_float2(p[j][0], p[j][1]);
          *reinterpret_cast<float2*>(to + 256 + 8 * j) = make_float2(p[j][2], p[j][3]);
        }
      }
      __syncthreads();
#pragma unroll 1
      for (int i = warp; i < cg * 16; i += NW) {             // a warp a row of a piece
        const int x = i >> 4, r = i & 15, pj = i0 + x;
        if (pj >= pairs) break;
        const int t = quot(pj, ck), key = 32 * (pj - t * ck) + lane;
        float sum = 0.f;
        const float* p = s_p + (x * hw * 16 + r) * 32 + lane;
#pragma unroll 2
        for (int h = 0; h < hw; ++h) sum += p[512 * h];
        if (r < s_tile[t].y && key < L) abar[(s_tile[t].x + r) * L + key] = sum * invh;
      }
      __syncthreads();
    }
  };

  bool from_x = false;
  if (a.h0_far) {                                              // rows in host memory cross the link once
    const int nv = d >> 3;
#pragma unroll 1
    for (int i = tid; i < mt * nv; i += NT) {
      const int t = quot(i, nv), at = 8 * (i - t * nv);        // CTA r copies row r of each tile
      const int4 tile = s_tile[t];
      if (rank < tile.y) *reinterpret_cast<uint4*>(a.x + (tile.x + rank) * d + at) =
          *reinterpret_cast<const uint4*>(a.h0 + (tile.z * L + (s_pos[16 * t + rank] & kPosMask)) * d + at);
    }
    cluster_arrive(); cluster_wait();
    from_x = true;
  }

  int lm_n = 0;
#pragma unroll 1
  for (int si = 0; si <= 4 * n_layers; ++si) {
    const int l = min(si >> 2, n_layers - 1), step = si == 4 * n_layers ? (int)S_LM : si & 3;
    bf16* kc = a.kc + (size_t)l * a.cache_layer; bf16* vc = a.vc + (size_t)l * a.cache_layer;
    const int tiles = step == S_LM ? (lm_n + 15) >> 4 : mt;
    const bool gathers = si == 0 && !from_x, normed = step != S_O && step != S_DOWN;
    // passes of as many tiles each as there are, up to P or what fits; rows of bf16, 64 bytes more apart than they are long
    const int sa = 2 * K + 64, most = min(P, quot(kPassBytes, RT * 4 + 16 * sa));
    const int passes = tiles > most ? quot(tiles + most - 1, most) : 1, pt = passes > 1 ? quot(tiles + passes - 1, passes) : tiles;
    unsigned char* s_act = reinterpret_cast<unsigned char*>(red + pt * RT);
#pragma unroll 1
    for (int p0 = 0; p0 < tiles; p0 += pt) {
      const int nt = min(pt, tiles - p0), nv = K >> 3;
      // What the epilogue reads from memory beside the sums, for the first of a thread's elements, which are two columns of lo and the
      // two of hi that belong to them, in a row of one (tile, unit) pair; 64 threads a pair.
      const int ec = (tid & 3) * 2, er = (tid >> 2) & 15;
      // ---- the rows' activations into shared memory ----------------------------------------------------
      const bf16* base = step == S_O ? a.o : step == S_DOWN ? a.hmid : gathers ? a.h0 : a.x;
#pragma unroll 1
      for (int i = warp; i < 16 * nt; i += NW) {
        int slot = 16 * p0 + i;
        if (step == S_LM) slot = slot < lm_n ? s_lm[slot] : -1;
        if (slot < 0 || (slot & 15) >= s_tile[slot >> 4].y) continue;
        const int4 tile = s_tile[slot >> 4];
        const bf16* p = base + (gathers ? tile.z * L + (s_pos[slot] & kPosMask) : tile.x + (slot & 15)) * K + 8 * lane;
        unsigned char* to = s_act + i * sa + 16 * lane;
#pragma unroll 1
        for (int c = lane; c < nv; c += 32, p += 256, to += 512) copy16(to, p);
      }
      if (step == S_O && p0 == 0 && l < a.depth) probabilities(l, kc);
      copies_done();
      __syncthreads();
      if (normed) {                                            // in place, half a warp a row
        const int hl = lane & 15;
#pragma unroll 1
        for (int i = 2 * warp + (lane >> 4); i < 16 * nt; i += 2 * NW) {
          uint4* at = reinterpret_cast<uint4*>(s_act + i * sa) + hl;
          const uint4* gain = reinterpret_cast<const uint4*>(s_gain) + hl;
          float ss = 0.f;
#pragma unroll 2
          for (int c = hl; c < nv; c += 16) {
            const uint4 x = at[c - hl];
            const float2 e = unpack2(x.x), f = unpack2(x.y), g = unpack2(x.z), h = unpack2(x.w);
            ss += (e.x * e.x + e.y * e.y + f.x * f.x + f.y * f.y) + (g.x * g.x + g.y * g.y + h.x * h.x + h.y * h.y);
          }
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
          const float rs = rsqrtf(__fdividef(ss, (float)d) + a.eps);
          bf16* also = nullptr;                                // who else wants the row as it was
          if (step == S_QKV && rank < 2) {
            const int slot = 16 * p0 + i;
            const int4 tile = s_tile[slot >> 4];
            if ((slot & 15) < tile.y) {
              const int row = tile.x + (slot & 15);
              if (gathers && rank == 0) also = a.x + row * d + 8 * hl;
              else if (rank == 1 && a.layer_in) also = a.layer_in + ((size_t)l * a.rows_cap + row) * d + 8 * hl;
            }
          }
#pragma unroll 2
          for (int c = hl; c < nv; c += 16) {
            const uint4 x = at[c - hl], gn = gain[c - hl];
            if (also) *reinterpret_cast<uint4*>(also + 8 * (c - hl)) = x;
            uint4 o;
            float2 f, g;
            f = unpack2(x.x); g = unpack2(gn.x); o.x = pack2(f.x * rs * g.x, f.y * rs * g.y);
            f = unpack2(x.y); g = unpack2(gn.y); o.y = pack2(f.x * rs * g.x, f.y * rs * g.y);
            f = unpack2(x.z); g = unpack2(gn.z); o.z = pack2(f.x * rs * g.x, f.y * rs * g.y);
            f = unpack2(x.w); g = unpack2(gn.w); o.w = pack2(f.x * rs * g.x, f.y * rs * g.y);
            at[c - hl] = o;
          }
        }
        __syncthreads();
      }
#pragma unroll 1
      for (int g = 0; g < units; g += per) {
        const int ng = min(units - g, per);
        int et = 0, eu = tid >> 6;
#pragma unroll 1
        while (eu >= ng) { eu -= ng; ++et; }
        uint32_t x0 = 0, x1 = 0;
        const bool first = et < nt && er < s_tile[p0 + et].y;
        if (!normed && first) {
          const bf16* x = a.x + (s_tile[p0 + et].x + er) * d + 16 * (u0 + g + eu) + ec;
          x0 = __ldcg(reinterpret_cast<const uint32_t*>(x)); x1 = __ldcg(reinterpret_cast<const uint32_t*>(x + 8));
        }
        // ---- the product -------------------------------------------------------------------------------
        if (ul < ng) {
          if (g + p0 > 0 && (per < units || nb > CB)) request(step, g);             // (otherwise it is still there)
#pragma unroll 1
          for (int b = 0; b < nb; b += CB) {
            if (b > 0) load_blocks(b);
            const unsigned char* p = s_act + g8 * sa + 16 * q;
#pragma unroll 1
            for (int t = 0; t < nt; ++t, p += 16 * sa) {
              float acc[2][2][4] = {};                         // [lo, hi][every other block]
#pragma unroll
              for (int j = 0; j < CB; j += 4) {
                if (b + j < nb) {                              // four blocks at a time; those that are not there weigh nothing
#pragma unroll
                  for (int i = j; i < j + 4; ++i) {
                    const unsigned char* at = p + 64 * (b0 + min(b + i, nb - 1));
                    const uint4 x = *reinterpret_cast<const uint4*>(at), z = *reinterpret_cast<const uint4*>(at + 8 * sa);
                    mma_k32(acc[0][i & 1], x, z, lo[i]);
                    mma_k32(acc[1][i & 1], x, z, hi[i]);
                  }
                }
              }
              float* to = red + (t * NW + warp) * 256 + g8 * 16;
#pragma unroll
              for (int h = 0; h < 2; ++h) {         // (halves of a row change places every second row: no bank twice)
                float2* r0 = reinterpret_cast<float2*>(to + ((8 * h + 2 * q) ^ (((g8 >> 1) & 1) << 3)));
                float2 v0 = make_float2(acc[h][0][0] + acc[h][1][0], acc[h][0][1] + acc[h][1][1]), v1 = make_float2(acc[h][0][2] + acc[h][1][2], acc[h][0][3] + acc[h][1][3]);
                if (b > 0) { v0.x += r0[0].x; v0.y += r0[0].y; v1.x += r0[64].x; v1.y += r0[64].y; }
                r0[0] = v0; r0[64] = v1;
              }
            }
          }
        }
        __syncthreads();
        // ---- epilogues ---------------------------------------------------------------------------------
        const int ks = 1 << lks;
        if (step != S_LM) {
          bool held = true;
#pragma unroll 1
          for (; et < nt; held = false) {
            const int4 tile = s_tile[p0 + et];
            if (er < tile.y) {
              const int sw = ((er >> 1) & 1) << 3, row = tile.x + er;
              const float* p = red + (et * NW + eu * ks) * 256 + er * 16;
              float2 vl = make_float2(0.f, 0.f), vh = make_float2(0.f, 0.f);
#pragma unroll 2
              for (int k = 0; k < ks; ++k, p += 256) {
                const float2 f = *reinterpret_cast<const float2*>(p + (ec ^ sw)), h = *reinterpret_cast<const float2*>(p + ((ec + 8) ^ sw));
                vl.x += f.x; vl.y += f.y; vh.x += h.x; vh.y += h.y;
              }
              const int U = u0 + g + eu;
              bf16 *to, *to2;
              if (step == S_QKV) {
                const int head = U / UH, at = 8 * (U - head * UH) + ec, pos = s_pos[16 * (p0 + et) + er] & kPosMask;
                if (a.layer[l].bqkv) {
                  const bf16* bias = a.layer[l].bqkv + head * DH + at;
                  const float2 bl = unpack2(__ldg(reinterpret_cast<const uint32_t*>(bias))), bh = unpack2(__ldg(reinterpret_cast<const uint32_t*>(bias + DH / 2)));
                  vl.x += bl.x; vl.y += bl.y; vh.x += bh.x; vh.y += bh.y;
                }
                if (head < hq + a.hkv) {
                  const float4 cs = __ldg(reinterpret_cast<const float4*>(a.rope + pos * (DH / 2) + at));
                  const float2 l2 = vl, h2 = vh;
                  vl = make_float2(l2.x * cs.x - h2.x * cs.y, l2.y * cs.z - h2.y * cs.w);
                  vh = make_float2(h2.x * cs.x + l2.x * cs.y, h2.y * cs.z + l2.y * cs.w);
                }
                if (head < hq) to = a.q + row * d_o + head * DH;
                else if (head < hq + a.hkv) to = kc + (tile.w + pos) * kv_ld + (head - hq) * DH;
                else to = vc + (tile.w + pos) * kv_ld + (head - hq - a.hkv) * DH;
                to += at; to2 = to + DH / 2;
              } else if (step == S_GATEUP) {
                vl = make_float2(__fdividef(vl.x, 1.f + __expf(-vl.x)) * vh.x, __fdividef(vl.y, 1.f + __expf(-vl.y)) * vh.y);
                to = a.hmid + row * a.ffn + 8 * U + ec; to2 = nullptr;
              } else {
                to = a.x + row * d + 16 * U + ec; to2 = to + 8;
                if (!held) { x0 = __ldcg(reinterpret_cast<const uint32_t*>(to)); x1 = __ldcg(reinterpret_cast<const uint32_t*>(to2)); }
                const float2 f = unpack2(x0), h = unpack2(x1);
                vl.x += f.x; vl.y += f.y; vh.x += h.x; vh.y += h.y;
              }
              *reinterpret_cast<uint32_t*>(to) = pack2(vl.x, vl.y);
              if (to2) *reinterpret_cast<uint32_t*>(to2) = pack2(vh.x, vh.y);
            }
            eu += NT / 64;
#pragma unroll 1
            while (eu >= ng) { eu -= ng; ++et; }
          }
        } else {
#pragma unroll 1
          for (int r = warp; r < 16 * nt && 16 * p0 + r < lm_n; r += NW) {           // a warp a row
            const int lm = s_lmlo + 16 * p0 + r;
            float mx = g == 0 ? -INFINITY : s_mx[r], sum = g == 0 ? 0.f : s_sum[r];
            int arg = g == 0 ? 0x7fffffff : s_arg[r];
            // (this warp's columns of the group, 32 at a time: running maximum and sum in every lane)
#pragma unroll 1
            for (int i0 = 0; i0 < 16 * ng; i0 += 32) {
              const int i = min(i0 + lane, 16 * ng - 1), c = i & 15, col = 16 * (u0 + g) + i;
              const float* p = red + ((r >> 4) * NW + (i >> 4) * ks) * 256 + (r & 15) * 16 + (c ^ (((r >> 1) & 1) << 3));
              float v = 0.f;
#pragma unroll 2
              for (int x = 0; x < ks; ++x) v += p[x * 256];
              const bool in = col < a.vocab && i == i0 + lane;
              if (a.logits && in) a.logits[lm * a.vocab + col] = v;
              float m = in ? v : -INFINITY;
              int at = in && v > -INFINITY ? col : 0x7fffffff;
              if (!(m >= -INFINITY)) m = -INFINITY;            // (not a number: never the maximum, but in the sum)
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, m, o);
                const int oa = __shfl_xor_sync(0xffffffffu, at, o);
                if (om > m || (om == m && oa < at)) { m = om; at = oa; }
              }
              const float top = fmaxf(mx, m);
              float e = in && v != -INFINITY ? __expf(v - top) : 0.f;
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
              sum = (mx == -INFINITY ? sum : sum * __expf(mx - top)) + e;
              if (m > mx) { mx = m; arg = at; }
            }
            if (lane == 0) {
              if (g + per >= units) a.lm_stats[lm * CL + rank] = make_float4(mx, __int_as_float(arg), sum, 0.f);
              else { s_mx[r] = mx; s_arg[r] = arg; s_sum[r] = sum; }
            }
            __syncwarp();
          }
        }
        if (g + per < units || p0 + pt < tiles) __syncthreads();
      }
    }
    if (step == S_LM) break;

    if (step == S_QKV) {
      grid.arrive();
      if (si == 0) { publish_rows(); __syncthreads(); lm_n = min(s_lmn, MAXT * 16); }
      grid.wait(61);
      // ---- attention of the cluster's rows over all keys: a CTA's warps share the units of a round, 16 keys at a time -----
      constexpr int SO = DH + 4;
      float* so = red;                                         // [warp][16][SO]
      float2* sml = reinterpret_cast<float2*>(so + NW * 16 * SO);       // [warp][16]
#pragma unroll 1
      for (int u = ua; u < ub; u += NW) {
        const int nr = min(NW, ub - u), lws = 3 - (nr > 1 ? 32 - __clz(nr - 1) : 0), ws = 1 << lws, un = warp >> lws, split = warp & (ws - 1);
        if (un < nr) {
          const int t = quot(u + un, hq), h = u + un - t * hq, kvh = quot(h, group);
          const int4 tile = s_tile[t];
          const bf16* kb = kc + tile.w * kv_ld + kvh * DH + 8 * q;
          const bf16* vb = vc + tile.w * kv_ld + kvh * DH + 8 * g8;
          const bf16* qp = a.q + tile.x * d_o + h * DH + 8 * q;
          const int stride = 16 * ws;
          int k0 = 16 * split;
          uint4 kf[2][DH / 32], v[4], qx[DH / 32], qy[DH / 32];
          auto load_k = [&](int at) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const bf16* kp = kb + min(at + 8 * j + g8, L - 1) * kv_ld;
#pragma unroll
              for (int i = 0; i < DH / 32; ++i) kf[j][i] = ldcg16(kp + 32 * i);
            }
          };
          auto load_v = [&](int at) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[i] = ldcg16(vb + min(at + 2 * q + (i & 1) + 8 * (i >> 1), L - 1) * kv_ld);
            }
          };
          {
            const bf16 *px = qp + min(g8, tile.y - 1) * d_o, *py = qp + min(g8 + 8, tile.y - 1) * d_o;
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) { qx[i] = ldcg16(px + 32 * i); qy[i] = ldcg16(py + 32 * i); }
          }
          load_k(k0); load_v(k0);
          float o[8][4], m0 = kNoKey, m1 = kNoKey, l0 = 0.f, l1 = 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
#pragma unroll 1
          for (; k0 < L; k0 += stride) {
            float s[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              s[j][0] = s[j][1] = s[j][2] = s[j][3] = 0.f;
#pragma unroll
              for (int i = 0; i < DH / 32; ++i) mma_k32(s[j], qx[i], qy[i], kf[j][i]);
            }
            const bool more = k0 + stride < L;
            if (more) load_k(k0 + stride);                     // (into the registers that the scores have just read)
            float mx0 = m0, mx1 = m1;
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                s[j][e] = k0 + 8 * j + 2 * q + (e & 1) < L ? s[j][e] * sc : -INFINITY;
                if (e < 2) mx0 = fmaxf(mx0, s[j][e]); else mx1 = fmaxf(mx1, s[j][e]);
              }
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
            const float c0 = ex2(m0 - mx0), c1 = ex2(m1 - mx1);
            m0 = mx0; m1 = mx1;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              s[j][0] = ex2(s[j][0] - m0); s[j][1] = ex2(s[j][1] - m0); s[j][2] = ex2(s[j][2] - m1); s[j][3] = ex2(s[j][3] - m1);
            }
            l0 = l0 * c0 + (s[0][0] + s[0][1] + s[1][0] + s[1][1]);
            l1 = l1 * c1 + (s[0][2] + s[0][3] + s[1][2] + s[1][3]);
            const uint32_t pa[4] = {pack2(s[0][0], s[0][1]), pack2(s[0][2], s[0][3]), pack2(s[1][0], s[1][1]), pack2(s[1][2], s[1][3])};
            // column g of product i is element 8 g + i of the head: neighbouring elements of a lane's four rows
            const uint32_t r[4][4] = {{v[0].x, v[0].y, v[0].z, v[0].w}, {v[1].x, v[1].y, v[1].z, v[1].w},
                                      {v[2].x, v[2].y, v[2].z, v[2].w}, {v[3].x, v[3].y, v[3].z, v[3].w}};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              o[i][0] *= c0; o[i][1] *= c0; o[i][2] *= c1; o[i][3] *= c1;
              const uint32_t pick = (i & 1) ? 0x7632 : 0x5410;
              mma16816(o[i], pa[0], pa[1], pa[2], pa[3], __byte_perm(r[0][i >> 1], r[1][i >> 1], pick), __byte_perm(r[2][i >> 1], r[3][i >> 1], pick));
            }
            if (more) load_v(k0 + stride);
          }
          l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
          l0 += __shfl_xor_sync(0xffffffffu, l0, 2); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
          if (q == 0) { sml[warp * 16 + g8] = make_float2(m0, l0); sml[warp * 16 + g8 + 8] = make_float2(m1, l1); }
          float* to = so + (warp * 16 + g8) * SO + 16 * q;
#pragma unroll
          for (int e = 0; e < 4; ++e)                          // c0, c1: row g; c2, c3: row g + 8
#pragma unroll
            for (int i = 0; i < 8; i += 4)
              *reinterpret_cast<float4*>(to + 8 * (e >> 1) * SO + 8 * (e & 1) + i) = make_float4(o[i][e], o[i + 1][e], o[i + 2][e], o[i + 3][e]);
        }
        __syncthreads();
        // a row's splits, side by side in a warp: the factor of each
        if ((tid >> lws) < nr * 16) {
          const int s = tid & (ws - 1), pr = tid >> lws, x = pr >> 4, r = pr & 15, at = (x * ws + s) * 16 + r;
          const float2 ml = sml[at];
          const unsigned act = __activemask();
          float m = ml.x;
#pragma unroll 1
          for (int o = 1; o < ws; o <<= 1) m = fmaxf(m, __shfl_xor_sync(act, m, o));
          const float f = ex2(ml.x - m);
          float sum = ml.y * f;
#pragma unroll 1
          for (int o = 1; o < ws; o <<= 1) sum += __shfl_xor_sync(act, sum, o);
          s_f[at] = __fdividef(f, sum);
          const int t = quot(u + x, hq);
          if (s == 0 && r < s_tile[t].y) a.lse[(s_tile[t].x + r) * hq + (u + x - t * hq)] = (m + __log2f(sum)) * kLn2;
        }
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < nr * 16 * (DH / 4); i += NT) {
          const int c = 4 * (i % (DH / 4)), r = i / (DH / 4) % 16, x = i / (DH / 4) / 16;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          const float* p = so + (x * ws * 16 + r) * SO + c;
          const float* pf = s_f + x * ws * 16 + r;
#pragma unroll 2
          for (int s = 0; s < ws; ++s, p += 16 * SO, pf += 16) {
            const float f = *pf;
            const float4 w = *reinterpret_cast<const float4*>(p);
            v.x += w.x * f; v.y += w.y * f; v.z += w.z * f; v.w += w.w * f;
          }
          const int t = quot(u + x, hq), h = u + x - t * hq;
          if (r < s_tile[t].y) *reinterpret_cast<uint2*>(a.o + (s_tile[t].x + r) * d_o + h * DH + c) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
        }
        if (u + NW < ub) __syncthreads();
      }
    }
    cluster_arrive();
    // ---- the next product's weights, then the barrier behind which its activations are ----------------------------------
    begin(si + 1 == 4 * n_layers ? (int)S_LM : (si + 1) & 3, min((si + 1) >> 2, n_layers - 1));
    cluster_wait();
    // ---- rollout (Eq. 6-9): the last layer's sums, which meet while the LM head runs -----------------------------------
    if (si == 4 * n_layers - 1 && a.depth == 1) { rollout_sums(0); grid.arrive(); }
  }

  // ---- Eq. 1 from the CTAs' maxima and sums ---------------------------------------------------------
  if (units == 0)
#pragma unroll 1
    for (int i = tid; i < lm_n; i += NT) a.lm_stats[(s_lmlo + i) * CL + rank] = make_float4(-INFINITY, __int_as_float(0x7fffffff), 0.f, 0.f);
  cluster_arrive(); cluster_wait();
#pragma unroll 1
  for (int at = rank + CL * warp; at < lm_n; at += CL * NW) {
    float4 st = make_float4(-INFINITY, __int_as_float(0x7fffffff), 0.f, 0.f);
    if (lane < CL) st = __ldcg(&a.lm_stats[(s_lmlo + at) * CL + lane]);
    float mx = st.x; int arg = __float_as_int(st.y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, mx, o);
      const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
      if (om > mx || (om == mx && oa < arg)) { mx = om; arg = oa; }
    }
    float sum = st.z == 0.f && mx != -INFINITY ? 0.f : st.z * __expf(st.x - mx);        // (a CTA without columns has nothing; not a number stays one)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
      const int s = s_lm[at], to = s_tile[s >> 4].z * L + (s_pos[s] & kPosMask);
      a.conf[to] = 1.f / sum; a.pred[to] = arg;
    }
  }
  // ---- the rest of the rollout, a layer at a time ------------------------------------------------------
#pragma unroll 1
  for (int l = a.depth - 1; l >= 0; --l) {
    if (a.depth > 1) {
      __syncthreads();
      rollout_sums(l);
      grid.arrive();
    }
    grid.wait(62);
    if (l > 0)
#pragma unroll 1
      for (int i = tid; i < mt * 16; i += NT) {
        const int4 t = s_tile[i >> 4];
        if ((i & 15) < t.y) s_u[i] = 0.5f * s_u[i] + 0.5f * sum_over_clusters(l, t.z, s_pos[i] & kPosMask);
      }
  }
#pragma unroll 1
  for (int i = blockIdx.x * NT + tid; i < B * L; i += gridDim.x * NT) {
    const int b = quot(i, L), j = i - b * L;
    if (s_off[b + 1] <= s_off[b]) continue;                    // a sequence without rows keeps its scores
    const float keep = __ldcg(a.sel.slot_of_pos + i) >= 0 ? 0.5f : 1.f;
    float v = 1.f;
#pragma unroll 1
    for (int l = a.depth - 1; l >= 0; --l) v = v * keep + 0.5f * sum_over_clusters(l, b, j);
    a.c[i] = v;
  }
  // The last CTA to leave clears the counters, also behind a wait that gave up: the next step finds them at zero.
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.sync + 1, 1u) == gridDim.x - 1) { a.sync[0] = 0; a.sync[1] = 0; }
  }
}

void config(int clusters, cudaStream_t st, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  cfg->gridDim = dim3(clusters * CL); cfg->blockDim = dim3(NT); cfg->dynamicSmemBytes = kSmallSmem; cfg->stream = st;
  attr[0].id = cudaLaunchAttributeCooperative; attr[0].val.cooperative = 1;
  cfg->attrs = attr; cfg->numAttrs = 1;
}
}  // namespace

// Asked for by every context when it is made, which sets the attributes that its launches need: kept from the first time on, one thread
// would find them done that another is only about to set, and take the refusal for the answer.
int small_step_clusters() {
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  config(1, nullptr, &cfg, attr);
  if (cudaFuncSetAttribute(small_step_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(small_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, small_step_kernel, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
  return n;
}

size_t small_step_scratch(const SmallArgs& a, int clusters, float* base, SmallArgs* out) {
  const size_t BL = (size_t)a.sel.batch * a.sel.seq_len;
  size_t at = 0;
  auto take = [&](size_t floats) { float* p = base + at; at += (floats + 63) / 64 * 64; return p; };
  float* lm = take(BL * CL * 4);
  float* rp = take((size_t)a.depth * clusters * BL);
  if (out) { out->lm_stats = reinterpret_cast<float4*>(lm); out->rp = rp; }
  return at;
}

int launch_small_step(const SmallArgs& a, int clusters, cudaStream_t st, bool* refused) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  config(clusters, st, &cfg, attr);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, small_step_kernel, a);
  // (what says that so many clusters do not fit here together, and nothing about the work before)
  *refused = e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported;
  if (*refused) { (void)cudaGetLastError(); return D2C_OK; }
  D2C_CUDA_OK(e);
  count_launch(1);
  return D2C_OK;
}

}  // namespace d2c

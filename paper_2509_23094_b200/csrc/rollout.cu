// Attention rollout influence scores (Eq. 6-9) without the L x L matrices.
//
// c^T = 1^T W^(N) ... W^(1).  A row of W^(l) is e_i for an unselected position and (Abar_i + e_i)/2
// for a selected one (Abar rows sum to 1, so the row sum of Eq. 7 is 2).  Evaluated from the left
// this is one vector-matrix product per layer, last layer first:
//     u'_j = u_j * (j selected ? 1/2 : 1) + 1/2 * sum_{i selected} u_i * Abar^(l)[i][j]
// The column sums stream Abar once (HBM-bound); rows are split across CTAs and the partial sums are
// added in a fixed order, so the result is deterministic.
//
// The chain is serial, so what a layer costs beside its bytes counts N times.  Up to 4 MB per layer and sequence one launch
// does it all: a cluster of eight CTAs per sequence holds u in shared memory, each CTA sums its eighth of the columns (the
// loads of a layer's first rows are in flight before the exchange that ends the layer before it) and writes its part of the
// new u to all eight.  It is bound by what eight SMs can read (about 100 GB/s each) and 2 us of exchange a layer: 32 layers of
// 768 columns take 68 us at 81 rows and 157 us at 489 (two launches a layer, which larger ones still take: 258 and 218 us,
// in the way of the projections that ran beside them); 8 layers of 1024 x 1024 72 and 75 us, where the line is drawn.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace d2c {
namespace {

__global__ void rollout_init_kernel(RolloutArgs a, uint8_t* insel) {
  pdl_prologue();
  const int b = blockIdx.y, L = a.seq_len;
  const int ro = a.row_off[b], nb = a.row_off[b + 1] - ro;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < L; j += gridDim.x * blockDim.x) {
    a.u0[(size_t)b * L + j] = 1.f;
    insel[(size_t)b * L + j] = 0;
  }
  __syncthreads();
  // the grid covers every position once, so each CTA marks the selected positions inside the
  // range it has just cleared
  const int j0 = blockIdx.x * blockDim.x, j1 = min(L, j0 + (int)blockDim.x);
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    const int pos = a.sel_idx[ro + i];
    if (pos >= j0 && pos < j1) insel[(size_t)b * L + pos] = 1;
  }
}

__global__ void __launch_bounds__(256)
rollout_partial_kernel(RolloutArgs a, const float* __restrict__ abar_l, const float* __restrict__ u) {
  pdl_prologue();
  const int b = blockIdx.z, s = blockIdx.y, L = a.seq_len;
  const int j = blockIdx.x * 256 + threadIdx.x;
  const int ro = a.row_off[b], nb = a.row_off[b + 1] - ro;
  if (nb <= 0) return;
  const int per = (nb + a.n_split - 1) / a.n_split;
  const int i0 = s * per, i1 = min(nb, i0 + per);
  float acc = 0.f;
  if (j < L) {
    const float* ub = u + (size_t)b * L;
    for (int i = i0; i < i1; ++i) {
      const float ui = ub[a.sel_idx[ro + i]];
      acc += ui * abar_l[(size_t)(ro + i) * L + j];
    }
    a.partial[((size_t)s * a.batch + b) * L + j] = acc;
  }
}

__global__ void __launch_bounds__(256)
rollout_combine_kernel(RolloutArgs a, const uint8_t* __restrict__ insel, const float* __restrict__ u,
                       float* __restrict__ out) {
  pdl_prologue();
  const int b = blockIdx.y, L = a.seq_len;
  const int j = blockIdx.x * 256 + threadIdx.x;
  if (j >= L || a.row_off[b + 1] - a.row_off[b] <= 0) return;
  float sum = 0.f;
  for (int s = 0; s < a.n_split; ++s) sum += a.partial[((size_t)s * a.batch + b) * L + j];
  const size_t o = (size_t)b * L + j;
  out[o] = u[o] * (insel[o] ? 0.5f : 1.f) + 0.5f * sum;
}

// ---- single launch ---------------------------------------------------------------------------
constexpr int kWarps = 16, kInFlight = 16;
// columns of a CTA, a multiple of four (a row's 16-byte pieces then start alike in every CTA)
__host__ __device__ inline int cluster_cols(int L) { return ((L + kRolloutCluster - 1) / kRolloutCluster + 3) & ~3; }
size_t cluster_smem(int L) { return ((size_t)3 * L + (size_t)kWarps * cluster_cols(L)) * sizeof(float) + cluster_cols(L); }

// Warp w sums the rows w, w + 16, ...: their distance is a multiple of four rows, so whatever L is, a row's first float
// lies at the same place of a 16-byte piece for all of a warp's rows, and lane q's piece holds the same four columns.
__global__ void __cluster_dims__(kRolloutCluster, 1, 1) __launch_bounds__(32 * kWarps, 1) rollout_cluster_kernel(RolloutArgs a) {
  pdl_prologue();
  extern __shared__ float sh[];
  const int b = blockIdx.y, L = a.seq_len, rank = (int)cluster_ctarank(), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ro = a.row_off[b], nb = a.row_off[b + 1] - ro;
  if (nb <= 0) return;                                         // (the same in all CTAs of the cluster)
  const long long total = (long long)a.row_off[a.batch] * L;   // floats of a layer that may be read
  const int step = cluster_cols(L), j0 = min(L, rank * step), cols = min(L, j0 + step) - j0;
  float* u[2] = {sh, sh + L};
  int* sel = reinterpret_cast<int*>(sh + 2 * L);
  float* part = sh + 3 * L;                                    // [warp][step]
  uint8_t* insel = reinterpret_cast<uint8_t*>(part + kWarps * step);
  for (int j = threadIdx.x; j < L; j += blockDim.x) u[0][j] = 1.f;
  for (int j = threadIdx.x; j < cols; j += blockDim.x) insel[j] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    const int pos = a.sel_idx[ro + i];
    sel[i] = pos;
    if (pos >= j0 && pos < j0 + cols) insel[pos - j0] = 1;
  }
  // a piece of work: up to kInFlight rows of a warp x its lanes' columns, 128 of them at a time
  const int n_rows = nb > warp ? (nb - warp + kWarps - 1) / kWarps : 0;
  int layer = a.n_layers - 1, r0 = 0, q0 = 0;                  // next piece: layer, first of the warp's rows, first 16-byte piece
  float4 x[kInFlight];
  int shift;                                                   // columns before j0 in the row's first 16-byte piece
  auto shift_of = [&](int l) {
    const float* p = a.abar + (size_t)l * a.layer_stride + (size_t)(ro + warp) * L + j0;
    return (int)((reinterpret_cast<uintptr_t>(p) >> 2) & 3);
  };
  auto request = [&]() {
    const float* base = a.abar + (size_t)layer * a.layer_stride;
    shift = shift_of(layer);
    const int c = 4 * (q0 + lane) - shift;                     // column of the piece's first float, from j0 on
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) {
      const int i = r0 + k;
      x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < n_rows && c < cols) {
        const long long at = (long long)(ro + warp + kWarps * i) * L + j0 + c;
        if (at >= 0 && at + 4 <= total) x[k] = __ldcg(reinterpret_cast<const float4*>(base + at));
        else {                                                 // the ends of the layer's rows
          if (at >= 0 && at < total) x[k].x = __ldcg(base + at);
          if (at + 1 >= 0 && at + 1 < total) x[k].y = __ldcg(base + at + 1);
          if (at + 2 >= 0 && at + 2 < total) x[k].z = __ldcg(base + at + 2);
          if (at + 3 >= 0 && at + 3 < total) x[k].w = __ldcg(base + at + 3);
        }
      }
    }
  };
  request();
  __syncwarp();
  cluster_sync_all();                                          // the others have started; this CTA's arrays are set
  for (int l = a.n_layers - 1; l >= 0; --l) {
    const float* uc = u[(a.n_layers - 1 - l) & 1];
    float* un = u[(a.n_layers - l) & 1];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    while (layer == l) {
      const int c = 4 * (q0 + lane) - shift;
#pragma unroll
      for (int k = 0; k < kInFlight; ++k) {
        const int i = r0 + k;
        const float ui = i < n_rows ? uc[sel[warp + kWarps * i]] : 0.f;
        if (i < n_rows) { acc.x += ui * x[k].x; acc.y += ui * x[k].y; acc.z += ui * x[k].z; acc.w += ui * x[k].w; }
      }
      r0 += kInFlight;
      if (r0 >= n_rows) {                                      // these columns' rows are summed
        float* p = part + warp * step + c;
        if (c >= 0 && c < cols) p[0] = acc.x;
        if (c + 1 >= 0 && c + 1 < cols) p[1] = acc.y;
        if (c + 2 >= 0 && c + 2 < cols) p[2] = acc.z;
        if (c + 3 >= 0 && c + 3 < cols) p[3] = acc.w;
        acc = make_float4(0.f, 0.f, 0.f, 0.f);
        r0 = 0; q0 += 32;
        if (4 * q0 - shift >= cols) { q0 = 0; --layer; }
      }
      if (layer >= 0) request();
    }
    __syncthreads();
    for (int j = threadIdx.x; j < cols; j += blockDim.x) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) sum += part[w * step + j];
      const float v = uc[j0 + j] * (insel[j] ? 0.5f : 1.f) + 0.5f * sum;
      if (l == 0) {
        a.c[(size_t)b * L + j0 + j] = v;
      } else {
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(un + j0 + j);
#pragma unroll
        for (int r = 0; r < kRolloutCluster; ++r) {
          uint32_t to;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(r));
          asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to), "f"(v) : "memory");
        }
      }
    }
    __syncwarp();
    if (l > 0) cluster_sync_all();                             // u is whole everywhere; part and the old u may be written again
  }
}

}  // namespace

bool rollout_single(const RolloutArgs& a) {
  const long long rows = a.expect_rows > 0 ? a.expect_rows : (long long)a.batch * a.seq_len;
  return !a.spread && a.seq_len <= 8192 && a.batch <= 8 && rows * a.seq_len * 4 <= (4LL << 20) * a.batch;
}

namespace {
int launch_rollout_cluster(const RolloutArgs& a, cudaStream_t st) {
  const size_t smem = cluster_smem(a.seq_len);
  static PerDevice attr_set;
  if (attr_set.first()) D2C_CUDA_OK(cudaFuncSetAttribute(rollout_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(8192)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kRolloutCluster, a.batch); cfg.blockDim = dim3(32 * kWarps); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  if (a.begun) {
    attr[0].id = cudaLaunchAttributeLaunchCompletionEvent;
    attr[0].val.launchCompletionEvent.event = a.begun; attr[0].val.launchCompletionEvent.flags = 0;
  } else {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = 1;
  D2C_CUDA_OK(cudaLaunchKernelEx(&cfg, rollout_cluster_kernel, a));
  count_launch(1);
  return D2C_OK;
}
}  // namespace

int launch_rollout(const RolloutArgs& a, cudaStream_t st) {
  if (a.batch <= 0 || a.seq_len <= 0 || a.n_layers <= 0) return D2C_OK;
  if (rollout_single(a)) return launch_rollout_cluster(a, st);
  const int L = a.seq_len;
  uint8_t* insel = reinterpret_cast<uint8_t*>(a.partial + (size_t)a.n_split * a.batch * L);
  D2C_LAUNCH((rollout_init_kernel), dim3(ceil_div(L, 256), a.batch), 256, 0, st, a, insel);
  const float* u = a.u0;
  float* bufs[2] = {a.u1, a.u0};
  for (int l = a.n_layers - 1; l >= 0; --l) {
    float* out = (l == 0) ? a.c : bufs[(a.n_layers - 1 - l) & 1];
    D2C_LAUNCH((rollout_partial_kernel), dim3(ceil_div(L, 256), a.n_split, a.batch), 256, 0, st, a, a.abar + (size_t)l * a.layer_stride, u);
    D2C_LAUNCH((rollout_combine_kernel), dim3(ceil_div(L, 256), a.batch), 256, 0, st, a, insel, u, out);
    u = out;
  }
  return D2C_OK;
}

}  // namespace d2c

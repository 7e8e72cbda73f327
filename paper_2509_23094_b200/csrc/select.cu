// Two-stage token selection of d2Cache (Section 4.1-4.2; one sequence by one CTA: select_seq.cuh) and the compaction of the selected set.
#include "select_seq.cuh"

namespace d2c {

__global__ void __launch_bounds__(kSelThreads) select_kernel(SelectArgs a) {
  pdl_prologue();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  select_sequence<false, kSelThreads>(a, blockIdx.x, smem_raw);
}

// Turns the per-sequence ranks into global row numbers.
__global__ void __launch_bounds__(256) select_finalize_kernel(SelectArgs a) {
  pdl_prologue();
  const int b = blockIdx.y, L = a.seq_len;
  int off = 0, lmoff = 0;
  for (int bb = 0; bb < b; ++bb) { off += a.n_b[bb]; lmoff += a.nm_b[bb]; }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.row_off[b] = off; a.lm_off[b] = lmoff;
    if (b == a.batch - 1) {
      a.row_off[a.batch] = off + a.n_b[b]; a.lm_off[a.batch] = lmoff + a.nm_b[b];
      if (a.n_host) *a.n_host = off + a.n_b[b];
    }
  }
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < L; j += gridDim.x * blockDim.x) {
    const int rs = a.rank_s[(size_t)b * L + j];
    int slot = -1;
    if (rs >= 0) {
      slot = off + rs;
      a.sel_idx[slot] = j;
      a.row_seq[slot] = b;
      const int rl = a.rank_lm[(size_t)b * L + j];
      if (rl >= 0) a.lm_rows[lmoff + rl] = slot;
    }
    a.slot_of_pos[(size_t)b * L + j] = slot;
  }
}

int launch_select(const SelectArgs& a, cudaStream_t st) {
  if (a.batch <= 0) return D2C_OK;
  // a sequence of 65535 selected rows would overflow the packed 16-bit counters
  if (a.seq_len > 8192) { set_global_error("select: seq_len %d > 8192", a.seq_len); return D2C_ECAPACITY; }
  const size_t smem = (size_t)a.seq_len * 11;               // two 32-bit words and three flag bytes per position
  static PerDevice attr_set;
  if (attr_set.first()) {
    D2C_CUDA_OK(cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 8192 * 11));
  }
  D2C_LAUNCH((select_kernel), a.batch, kSelThreads, smem, st, a);
  if (a.batch > 1) {
    dim3 grid(ceil_div(a.seq_len, 256), a.batch);
    D2C_LAUNCH((select_finalize_kernel), grid, 256, 0, st, a);
  }
  return D2C_OK;
}

int build_phi_table(float sigma, uint32_t* tab, int len) {
  const double s = (double)sigma;
  int first_zero = len;
  for (int r = 0; r < len; ++r) {
    const double rr = (double)r;
    const double v = exp(-(rr * rr) / (2.0 * s * s)) * 1073741824.0;
    tab[r] = (uint32_t)floor(v + 0.5);
    if (tab[r] == 0 && first_zero == len) first_zero = r;
  }
  return first_zero;
}

}  // namespace d2c

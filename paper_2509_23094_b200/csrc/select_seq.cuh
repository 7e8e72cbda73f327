// Two-stage token selection of one sequence (Section 4.1-4.2) by one CTA: the body of the selection kernel and of the first phase of
// the kernel that does a small model's whole step.  To be compiled without fast math: indices are decided from fp32 products.
//
// One CTA per sequence.  Every sum that decides an index is an integer sum, so the result does
// not depend on the order in which threads add:
//   stage 1 (Eq. 3-4): D(i) = sum over known j of phi(|i-j|), with phi tabulated as round(phi*2^30);
//                      key = fp32(D) * conf (one multiply); the k largest keys among masked positions
//                      (equal keys: lower position first).
//   stage 2 (after Eq. 9): candidates in the order (score c_j descending, position ascending); the shortest
//                      prefix whose mass sum floor(c_j*2^32) exceeds p times the total.
// Neither stage sorts.  Both are "take elements in that order until a running weight crosses a threshold"
// (weight 1 and threshold k for stage 1, the fixed-point mass and p * total for stage 2), which needs only the
// score value at which the crossing happens: four 8-bit radix passes over the fp32 bit patterns, each a
// 256-bin histogram of weights scanned from the top, find it exactly; elements above that value are taken,
// elements equal to it are taken in position order while the running weight has not crossed.  Up to 1024
// masked positions (every decoding step of the workloads) stage 1 skips even that and ranks each masked
// position against all others directly, one position per thread.
#pragma once
#include <math.h>

#include "common.cuh"

namespace d2c {

static constexpr int kSelThreads = 512;
static constexpr int kPhiMax = 512;              // phi entries kept in shared memory; a wider window reads the rest from global memory
static constexpr int kRankMax = 1024;            // stage 1 ranks by direct comparison up to this many masked positions
static constexpr int kSumMax = 128;              // stage 2 sums by direct comparison up to this many candidates
enum : uint8_t { F_SEL = 1, F_MSTAR = 2 };

// Exclusive block scan of one value per thread; returns the exclusive prefix, *total gets the sum.
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* warp_buf, T* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T up = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += up;
  }
  if (lane == 31) warp_buf[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    T w = lane < nw ? warp_buf[lane] : T(0);
    T winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T up = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += up;
    }
    warp_buf[lane] = winc - w;                     // exclusive prefix of warp sums
    if (lane == 31) *total = winc;
  }
  __syncthreads();
  T res = warp_buf[wid] + inc - v;
  __syncthreads();
  return res;
}

// NaN, negative and infinite scores count as 0; finite ones are capped at 2^18 so that the fixed-point
// mass of 8192 positions stays inside 64 bits.
__device__ __forceinline__ float clean_score(float x) { return (x > 0.f && x < INFINITY) ? fminf(x, 262144.f) : 0.f; }

// Shared scratch of the threshold search.
struct RadixScratch {
  // per digit: the weight sum of the members that carry it, kept as three 32-bit sums of 17-bit pieces of the
  // weights (weights stay below 2^51, 8192 positions x 2^17 below 2^32): 32-bit shared-memory atomics are native,
  // the 64-bit ones took about seven clocks per lane whatever the address (6700 of a 1024-position pass's clocks)
  uint32_t hist[3][256];
  unsigned long long warp_buf[32];
  unsigned long long total;
  unsigned long long above;
  int digit;                               // crossing digit of the pass, -1: the weight of all members does not cross
  int few;                                 // members that carry the crossing digits so far; the first kFew of them:
  unsigned long long few_key[32], few_w[32];      // value bits << 32 | ~position, weight
};
constexpr int kFew = 32;

__device__ __forceinline__ unsigned long long shfl_up_u64(unsigned long long v, int o) {
  const uint32_t lo = __shfl_up_sync(0xffffffffu, (uint32_t)v, o), hi = __shfl_up_sync(0xffffffffu, (uint32_t)(v >> 32), o);
  return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long v, int o) {
  const uint32_t lo = __shfl_xor_sync(0xffffffffu, (uint32_t)v, o), hi = __shfl_xor_sync(0xffffffffu, (uint32_t)(v >> 32), o);
  return ((unsigned long long)hi << 32) | lo;
}

// The shortest prefix, in the order (value bits descending, position ascending), of the positions j < L with
// member(j) whose running weight "crosses": crossed(w) must be monotone in w and false for w = 0.  Sets `mark`
// in flags for every position of that prefix; if the weight never crosses, for every member.
// weight(bits) is 1 (counting) or the fixed-point mass; all members with equal bits have equal weight.
// rs.hist must be zero on entry and is zero again on return.
// [vmin, vmax] bounds the members' value bits.  Digits are taken from the distance to vmin, eight bits at a time from its
// highest on: the first pass spreads the members over up to 256 bins whatever their scale, and as soon as no more than 32 carry
// the crossing digits, one warp places those by comparing them with each other.  (A pass takes 2500 clocks, mostly latency.
// Flat scores of 1024 positions took three or four and now take one and that comparison: a step of 277 rows in two sequences
// 139.3 -> 135.7 us, one of 55 in 546 122.7 -> 120.7.)
template <typename Member, typename Weight, typename Crossed>
__device__ __forceinline__ void take_until_crossed(const uint32_t* vb, int L, Member member, Weight weight, Crossed crossed,
                                                   uint8_t* flags, uint8_t mark, RadixScratch& rs, uint32_t vmin, uint32_t vmax) {
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
  uint32_t pref = 0;                                     // the high digits fixed so far (of the distance to vmin)
  unsigned long long above = 0;                          // weight of the members above the range still searched
  bool all = false;
  int rem = max(32 - __clz(vmax - vmin), 1);             // bits not fixed yet
  bool first = true;
  while (rem > 0 && !all) {
    const int bits = min(rem, 8), shift = rem - bits;
    for (int base = 0; base < L; base += T) {
      const int j = base + tid;
      const uint32_t dist = j < L ? vb[j] - vmin : 0u;
      const bool m = j < L && member(j) && (first || (dist >> rem) == pref);
      const unsigned act = __ballot_sync(0xffffffffu, m);
      if (act) {
        // a warp whose live lanes all carry the same digit adds once; otherwise each lane adds
        const uint32_t d = m ? (dist >> shift) & ((1u << bits) - 1u) : 0u;
        unsigned long long w = m ? weight(vb[j]) : 0ull;
        const int leader = __ffs(act) - 1;
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, leader);
        const bool one_digit = __all_sync(0xffffffffu, !m || d == d0);
        if (one_digit)
          for (int o = 16; o > 0; o >>= 1) w += shfl_xor_u64(w, o);
        if (one_digit ? lane == leader : m) {
          // (a warp's sum of 32 weights may carry into bit 51 and above: the top piece takes all the high bits)
          const uint32_t w0 = (uint32_t)(w & 0x1FFFFull), w1 = (uint32_t)((w >> 17) & 0x1FFFFull), w2 = (uint32_t)(w >> 34);
          if (w0) atomicAdd(&rs.hist[0][d], w0);
          if (w1) atomicAdd(&rs.hist[1][d], w1);
          if (w2) atomicAdd(&rs.hist[2][d], w2);
        }
      }
    }
    __syncthreads();
    if (tid < 32) {
      // one warp walks the digits from the top: lane l owns digits 255 - 8 l down to 248 - 8 l
      unsigned long long w[8], sum = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int bin = 255 - (8 * lane + k);
        w[k] = (unsigned long long)rs.hist[0][bin] + ((unsigned long long)rs.hist[1][bin] << 17) + ((unsigned long long)rs.hist[2][bin] << 34);
        rs.hist[0][bin] = 0; rs.hist[1][bin] = 0; rs.hist[2][bin] = 0;
        sum += w[k];
      }
      unsigned long long inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long up = shfl_up_u64(inc, o);
        if (lane >= o) inc += up;
      }
      unsigned long long run = above + inc - sum;        // weight above this lane's first digit
      int hit = -1; unsigned long long before = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (hit < 0 && w[k] != 0 && crossed(run + w[k])) { hit = k; before = run; }
        run += w[k];
      }
      const unsigned found = __ballot_sync(0xffffffffu, hit >= 0);
      if (lane == 0) rs.few = 0;
      if (found == 0) {
        if (lane == 0) rs.digit = -1;
      } else if (lane == __ffs(found) - 1) {
        rs.digit = 255 - (8 * lane + hit);
        rs.above = before;
      }
    }
    __syncthreads();
    first = false;
    if (rs.digit < 0) {
      all = true;                                        // the weight of all members together does not cross
      break;
    }
    above = rs.above;
    pref = (pref << bits) | (uint32_t)rs.digit;
    rem = shift;
    for (int j = tid; j < L; j += T)
      if (member(j) && ((vb[j] - vmin) >> rem) == pref) {
        const int at = atomicAdd(&rs.few, 1);
        if (at < kFew) {
          rs.few_key[at] = ((unsigned long long)vb[j] << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)j);
          rs.few_w[at] = weight(vb[j]);
        }
      }
    __syncthreads();
    const int few = rs.few;
    if (few <= kFew) {
      // The members of higher digits are in; of these, those before which the weight has not crossed.
      for (int j = tid; j < L; j += T)
        if (member(j) && ((vb[j] - vmin) >> rem) > pref) flags[j] |= mark;
      if (tid < few) {
        const unsigned long long mine = rs.few_key[tid];
        unsigned long long before = above;
        for (int f = 0; f < few; ++f) before += rs.few_key[f] > mine ? rs.few_w[f] : 0ull;
        if (!crossed(before)) flags[0xFFFFFFFFu - (uint32_t)(mine & 0xFFFFFFFFull)] |= mark;
      }
      __syncthreads();
      return;
    }
    // (rs.digit and rs.few are rewritten only behind the next pass's barrier)
  }
  pref += vmin;                                          // the crossing value
  // members above the crossing value are in; those equal to it, in position order, while the weight before them has not crossed
  const int per = (L + T - 1) / T;
  const int j0 = tid * per;
  unsigned long long ties = 0;
  if (!all)
    for (int e = 0; e < per; ++e) {
      const int j = j0 + e;
      if (j < L && member(j) && vb[j] == pref) ++ties;
    }
  unsigned long long r = all ? 0ull : block_exclusive_scan<unsigned long long>(ties, rs.warp_buf, &rs.total);
  const unsigned long long wstar = weight(pref);
  for (int e = 0; e < per; ++e) {
    const int j = j0 + e;
    if (j >= L || !member(j)) continue;
    bool in = all || vb[j] > pref;
    if (!all && vb[j] == pref) { in = !crossed(above + r * wstar); ++r; }
    if (in) flags[j] |= mark;
  }
  __syncthreads();
}

// Selects the rows of sequence b, by a CTA of kThreads.  smem_raw: 11 bytes a position.  kOneKernel: the rest of the step is in the same kernel and works out the
// rows' global numbers itself, so all that is left here is rank_s[rank] = position | (rank among the masked + 1, 0: none) << kPosBits
// and slot_of_pos = -1 where nothing is selected.
constexpr int kPosBits = 13;
template <bool kOneKernel, int kThreads>
__device__ __forceinline__ void select_sequence(const SelectArgs& a, int b, unsigned char* smem_raw) {
  const int L = a.seq_len, tid = threadIdx.x, lane = tid & 31;
  uint32_t* kb = reinterpret_cast<uint32_t*>(smem_raw);       // stage-1 key bits (0 outside the stage-1 set)
  uint32_t* cb = kb + L;                                       // stage-2 score bits
  uint8_t* flags = reinterpret_cast<uint8_t*>(cb + L);
  uint8_t* smask = flags + L;
  uint8_t* in1 = smask + L;                                    // 1: masked and inside the block (the set stage 1 ranks)
  __shared__ RadixScratch rsc;
  __shared__ unsigned long long mlist[kRankMax];               // stage-1 members: position, then (key bits << 32 | ~position)
  __shared__ int warp_buf32[32];
  __shared__ int s_total32, s_nm, s_known, s_listed;
  __shared__ unsigned long long s_mass;
  __shared__ uint32_t s_lo, s_hi;
  __shared__ uint32_t s_phi[kPhiMax];                          // the non-zero head of the phi table (window +-65 at sigma 10)

  const uint8_t* mask = a.mask + (size_t)b * L;
  const float* conf = a.conf + (size_t)b * L;
  const float* cs = a.c + (size_t)b * L;
  const float* okey = a.override_key ? a.override_key + (size_t)b * L : nullptr;
  float* key_out = a.key + (size_t)b * L;

  int f0 = 0, n_forced = 0, first_forced = -1;                 // forced rows: the first of them is loaded long before it is needed (0.2 to 0.5 us)
  if (a.forced && a.forced_off) { f0 = a.forced_off[b]; n_forced = a.forced_off[b + 1] - f0; }

  // stage 1 may be confined to one block of positions (semi-autoregressive decoding); whole sequence otherwise
  const int blk_lo = a.block_hi > a.block_lo ? a.block_lo : 0, blk_hi = a.block_hi > a.block_lo ? a.block_hi : L;
  for (int i = tid; i < L; i += kThreads) {
    smask[i] = mask[i] ? 1 : 0; flags[i] = 0; kb[i] = 0;
    cb[i] = __float_as_uint(clean_score(cs[i]));
  }
  for (int r = tid; r < min(a.phi_len, kPhiMax); r += kThreads) s_phi[r] = a.phi_q30[r];
  for (int i = tid; i < 3 * 256; i += kThreads) (&rsc.hist[0][0])[i] = 0;
  if (tid == 0) { s_nm = 0; s_known = 0; s_listed = 0; s_mass = 0; s_lo = 0xFFFFFFFFu; s_hi = 0u; }
  __syncthreads();
  if (tid < n_forced) first_forced = a.forced[f0 + tid];

  // ---- the set stage 1 ranks: masked positions inside the block, listed in any order; known positions are counted ----
  int known = 0;
  for (int base = 0; base < L; base += kThreads) {
    const int i = base + tid;
    const bool m1 = i < L && smask[i] && i >= blk_lo && i < blk_hi;
    known += __popc(__ballot_sync(0xffffffffu, i < L && !smask[i]));
    if (i < L) { in1[i] = m1 ? 1 : 0; if (!m1) key_out[i] = 0.f; }
    const unsigned act = __ballot_sync(0xffffffffu, m1);
    if (act) {
      int slot0 = 0;
      if (lane == __ffs(act) - 1) slot0 = atomicAdd(&s_nm, __popc(act));
      slot0 = __shfl_sync(0xffffffffu, slot0, __ffs(act) - 1);
      const int slot = slot0 + __popc(act & ((1u << lane) - 1u));
      if (m1 && slot < kRankMax) mlist[slot] = (unsigned long long)i;
    }
  }
  if (lane == 0) atomicAdd(&s_known, known);
  __syncthreads();
  const int nm = s_nm, take = min(max(a.k, 0), nm);

  // ---- keys (Eq. 3-4): D(i) as an exact integer sum over the window, key = fp32(D) * confidence ----
  auto known_at = [&](int i, int r) {
    const int lo = i - r, hi = i + r;
    int known = 0;
    if (lo >= 0) known += 1 - smask[lo];
    if (hi < L) known += 1 - smask[hi];
    return (unsigned)known;
  };
  auto finish_key = [&](int i, unsigned long long dq, float cf) {
    float key;
    if (okey) {
      key = clean_score(okey[i]);
    } else {
      const float D = __ull2float_rn(dq) * 9.31322574615478515625e-10f;       // * 2^-30, exact
      key = clean_score(__fmul_rn(D, cf));
    }
    key_out[i] = key;
    kb[i] = __float_as_uint(key);
    return key;
  };
  if (nm <= kRankMax) {
    // a group of tpm lanes (a power of two, inside one warp) shares the window of one listed position
    int tpm = 1;
    while (tpm < 32 && 2 * tpm * nm <= kThreads) tpm <<= 1;
    const int sub = tid & (tpm - 1), groups = kThreads / tpm;
    for (int e0 = 0; e0 < nm; e0 += groups) {
      const int e = e0 + tid / tpm;
      const bool live = e < nm;
      const int i = live ? (int)mlist[e] : 0;
      const float cf = (live && sub == 0 && !okey) ? conf[i] : 0.f;       // in flight while the window is summed
      unsigned long long dq = 0;
      if (live && !okey)
        for (int r = 1 + sub; r < a.phi_len; r += tpm)
          dq += (unsigned long long)(r < kPhiMax ? s_phi[r] : a.phi_q30[r]) * known_at(i, r);
      for (int o = 1; o < tpm; o <<= 1) dq += shfl_xor_u64(dq, o);
      __syncwarp();
      if (live && sub == 0) {
        const float key = finish_key(i, dq, cf);
        mlist[e] = ((unsigned long long)__float_as_uint(key) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)i);
      }
    }
  } else {
    for (int i = tid; i < L; i += kThreads) {
      if (!in1[i]) continue;
      unsigned long long dq = 0;
      if (!okey)
        for (int r = 1; r < a.phi_len; ++r) dq += (unsigned long long)(r < kPhiMax ? s_phi[r] : a.phi_q30[r]) * known_at(i, r);
      finish_key(i, dq, okey ? 0.f : conf[i]);
    }
  }
  __syncthreads();

  // ---- stage 1: the k largest keys of the set, lower position first among equal keys ----
  {
    if (take == nm) {
      for (int i = tid; i < L; i += kThreads)
        if (in1[i]) flags[i] = F_SEL | F_MSTAR;
    } else if (take > 0 && nm <= kRankMax) {
      // rank of a listed position = how many others come before it; a group of tpe lanes (a power of two, inside
      // one warp) shares a position and each counts every tpe-th entry
      int tpe = 1;
      while (tpe < 32 && 2 * tpe * nm <= kThreads) tpe <<= 1;
      const int sub = tid & (tpe - 1), groups = kThreads / tpe;
      for (int e0 = 0; e0 < nm; e0 += groups) {
        const int e = e0 + tid / tpe;
        const bool live = e < nm;
        const unsigned long long mine = live ? mlist[e] : 0ull;
        int rank = 0;
        if (live)
          for (int f = sub; f < nm; f += tpe) rank += mlist[f] > mine ? 1 : 0;
        for (int o = 1; o < tpe; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (live && sub == 0 && rank < take) flags[0xFFFFFFFFu - (uint32_t)(mine & 0xFFFFFFFFull)] = F_SEL | F_MSTAR;
      }
    } else if (take > 0) {
      const unsigned long long want = (unsigned long long)take;
      take_until_crossed(kb, L, [&](int j) { return in1[j] != 0; }, [](uint32_t) { return 1ull; },
                         [&](unsigned long long w) { return w >= want; }, flags, (uint8_t)(F_SEL | F_MSTAR), rsc, 0u, 0xFFFFFFFFu);
    }
    __syncthreads();
  }

  // ---- stage 2: top-p over the candidates by influence score ----
  // (The loops from here on are hardly unrolled: a step's weights drive these instructions out of the caches, and what is not unrolled
  // need not come back.  The kernel alone, caches cold, 1024 positions: 19.5 -> 16.9 us; steps: three sequences of 701 positions 91.2 ->
  // 90.4 us, 94 rows of 128 59.7 -> 58.3 and 105.8 -> 105.1.)
  if (a.p > 0.f) {
    const bool mode1 = a.stage2_candidates != 0;
    auto cand = [&](int j) { return mode1 ? (flags[j] & F_MSTAR) == 0 : smask[j] == 0; };
    auto mass = [](uint32_t bits) { return (unsigned long long)__double2ull_rd((double)__uint_as_float(bits) * 4294967296.0); };
    unsigned long long local = 0;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    // Few candidates are listed, in any order, for the direct sums below (stage 1 is done with its list).  Only they: listing 500 to
    // 1500, of which none is looked at, took up to 1 us of a step.
    unsigned long long *ckey = mlist, *cmass = mlist + kSumMax;
    const int nc = mode1 ? L - take : s_known;
#pragma unroll 1
    for (int j = tid; j < L; j += kThreads)
      if (cand(j)) {
        const unsigned long long w = mass(cb[j]);
        local += w; lo = min(lo, cb[j]); hi = max(hi, cb[j]);
        if (nc <= kSumMax) {
          const int slot = atomicAdd(&s_listed, 1);
          ckey[slot] = ((unsigned long long)cb[j] << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)j); cmass[slot] = w;
        }
      }
    for (int o = 16; o > 0; o >>= 1) local += shfl_xor_u64(local, o);
    lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      if (local) atomicAdd(&s_mass, local);
      atomicMin(&s_lo, lo); atomicMax(&s_hi, hi);
    }
    __syncthreads();
    // (p above 1 selects every candidate, as p = 1 does: the total never exceeds itself)
    const double thr = __dmul_rn(fmin((double)a.p, 1.0), __ull2double_rn(s_mass));
    // The prefix's mass has crossed when double(mass) > thr.  double() is monotone, so that is mass >= T for the
    // smallest integer T whose double exceeds thr, and the search compares integers.  Below 2^52 every integer is
    // its own double: T = floor(thr) + 1; above, T lies within 2048 of floor(thr) (doubles are at most 1024 apart
    // below 2^63) and a bisection finds it.
    unsigned long long T;
    {
      const unsigned long long fl = __double2ull_rd(thr);
      if (thr < 4503599627370496.0) {
        T = fl + 1ull;
      } else {
        unsigned long long lo_t = fl - 2048ull, hi_t = fl + 2049ull;        // double(lo_t) <= thr < double(hi_t)
        while (hi_t - lo_t > 1ull) {
          const unsigned long long mid = lo_t + ((hi_t - lo_t) >> 1);
          if (__ull2double_rn(mid) > thr) hi_t = mid; else lo_t = mid;
        }
        T = hi_t;
      }
    }
    if (nc <= kSumMax) {
      // few candidates: the mass before each of them, a group of tpe lanes (a power of two, inside one warp) to a candidate.  A step of
      // the smallest model, us, this way / by digits: 96 candidates 53.2 / 53.9, 120 57.6 / 58.2, 128 57.4 / 57.7, 150 59.3 / 59.2, 180
      // 60.0 / 60.0, 210 62.3 / 61.4, 300 68.1 / 64.3.
      int tpe = 1;
      while (tpe < 32 && 2 * tpe * nc <= kThreads) tpe <<= 1;
      const int sub = tid & (tpe - 1), groups = kThreads / tpe;
      for (int e0 = 0; e0 < nc; e0 += groups) {
        const int e = e0 + tid / tpe;
        const unsigned long long mine = e < nc ? ckey[e] : 0ull;
        unsigned long long before = 0;
        if (e < nc)
#pragma unroll 2
          for (int f = sub; f < nc; f += tpe) before += ckey[f] > mine ? cmass[f] : 0ull;
        for (int o = 1; o < tpe; o <<= 1) before += shfl_xor_u64(before, o);
        if (e < nc && sub == 0 && before < T) flags[0xFFFFFFFFu - (uint32_t)(mine & 0xFFFFFFFFull)] |= F_SEL;
      }
      __syncthreads();
    } else {
      take_until_crossed(cb, L, cand, mass, [&](unsigned long long w) { return w >= T; }, flags, (uint8_t)F_SEL, rsc,
                         s_lo, max(s_hi, s_lo));
    }
  }

  // ---- forced rows ----
#pragma unroll 1
  for (int f = tid; f < n_forced; f += kThreads) {
    const int pos = f == tid ? first_forced : a.forced[f0 + f];
    if (pos >= 0 && pos < L) flags[pos] = flags[pos] | F_SEL;   // duplicates write the same value
  }
  __syncthreads();

  // ---- ranks of the selected positions (ascending) and of the selected masked positions ----
  {
    const int per = (L + kThreads - 1) / kThreads;
    const int j0 = tid * per;
    int local = 0;                                     // low 16 bits: selected, high 16: selected & masked
#pragma unroll 1
    for (int e = 0; e < per; ++e) {
      const int j = j0 + e;
      if (j < L && (flags[j] & F_SEL)) local += 1 + (smask[j] ? (1 << 16) : 0);
    }
    int excl = block_exclusive_scan<int>(local, warp_buf32, &s_total32);
#pragma unroll 1
    for (int e = 0; e < per; ++e) {
      const int j = j0 + e;
      if (j >= L) break;
      uint32_t r = 0xFFFFFFFFu;                        // low 16 bits: rank, high 16: rank among the masked (0xFFFF: none)
      if (flags[j] & F_SEL) {
        r = (uint32_t)(excl & 0xFFFF) | 0xFFFF0000u;
        if (smask[j]) { r = (uint32_t)excl; excl += 1 << 16; }
        excl += 1;
      }
      kb[j] = r;                                       // (the keys are not needed any more)
    }
    __syncthreads();
    // written position by position: neighbouring threads, neighbouring words (2048 positions 205.0 -> 203.3 us, up to 1024 no difference)
#pragma unroll 1
    for (int j = tid; j < L; j += kThreads) {
      const uint32_t r = kb[j];
      const int rs = r == 0xFFFFFFFFu ? -1 : (int)(r & 0xFFFFu), rl = rs < 0 || (r >> 16) == 0xFFFFu ? -1 : (int)(r >> 16);
      if (kOneKernel) {
        if (rs >= 0) a.rank_s[(size_t)b * L + rs] = j | ((rl + 1) << kPosBits);
        else a.slot_of_pos[(size_t)b * L + j] = -1;
      } else if (a.batch == 1) {
        // one sequence: its ranks are the global row numbers, so the second kernel's work is done here
        if (rs >= 0) {
          a.sel_idx[rs] = j; a.row_seq[rs] = 0;
          if (rl >= 0) a.lm_rows[rl] = rs;
        }
        a.slot_of_pos[j] = rs;
      } else {
        a.rank_s[(size_t)b * L + j] = rs;
        a.rank_lm[(size_t)b * L + j] = rl;
      }
    }
    if (tid == 0) { a.n_b[b] = s_total32 & 0xFFFF; a.nm_b[b] = s_total32 >> 16; }
    if (!kOneKernel && a.batch == 1) {
      if (tid == 0) {
        a.row_off[0] = 0; a.lm_off[0] = 0; a.row_off[1] = s_total32 & 0xFFFF; a.lm_off[1] = s_total32 >> 16;
        if (a.n_host) *a.n_host = s_total32 & 0xFFFF;
      }
    }
  }
}

}  // namespace d2c

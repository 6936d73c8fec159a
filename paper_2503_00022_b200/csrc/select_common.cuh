// Block-wide building blocks shared by the signature, the token-level and the page-level selection kernels:
// the search for the k-th largest key by radix histograms, exact top-k marking of 64-bit keys and emission of
// the kept set from two membership masks.
#pragma once

#include "common.cuh"

namespace kvc {
namespace sel {

constexpr int kMaxWarps = 32;                  // the helpers below take the block's thread count kT, at most 1024
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kDigitBits = 11;                 // radix digit of the 64-bit selection
constexpr int kBins = 1 << kDigitBits;
constexpr int kSmallList = 32;                 // 32-bit candidates one warp ranks directly
constexpr int kRankList = 256;                 // 64-bit candidates a block ranks directly, at most

struct Scratch {
  alignas(16) uint32_t hist[kBins];
  unsigned long long red[kMaxWarps];           // per-warp maximum and minimum of the keys' upper halves
  unsigned long long small[kRankList];
  unsigned long long sel_x;                    // result of a ranking
  uint32_t sel[3];                             // digit, remaining rank, live keys
  uint32_t small_n;
  int warp_tot[kMaxWarps];
};

__device__ __forceinline__ uint32_t head_mask(int Hq, int w) {
  const int n = Hq - 32 * w;
  return n >= 32 ? 0xFFFFFFFFu : ((1u << n) - 1u);
}

// Sum of tot[0 .. warp) for every thread of warp `warp`: one load per lane and a warp reduction instead of a serial
// walk (the last warp would otherwise do 31 dependent loads).  n_warps <= 32.
__device__ __forceinline__ int warps_before(const int* tot, int warp, int lane) {
  return __reduce_add_sync(kFull, lane < warp ? tot[lane] : 0);
}

// Contiguous item range of a warp: a multiple of 32 items, so that mask words do not straddle warps.
template <int kT>
__device__ __forceinline__ void warp_range(int n, int warp, int& r_lo, int& r_hi) {
  const int n_words = (n + 31) >> 5;
  const int per_warp = ((n_words + kT / 32 - 1) / (kT / 32)) * 32;
  r_lo = min(n, warp * per_warp);
  r_hi = min(n, r_lo + per_warp);
}

// The digit that holds the k_rem-th largest key, from a complete histogram of one digit position (bins in
// ascending digit order, counted from the top): out[0] = digit, out[1] = rank left inside that digit's bin,
// out[2] = keys in the bin.  Called by all kT threads of the block; k_rem is at most the histogram's total.
// The histogram must be complete (a barrier lies between its last update and this call); the result is
// visible to every thread on return.
template <int kT>
__device__ __forceinline__ void find_digit_desc(const uint32_t* hist, int n_bins, uint32_t k_rem, int* warp_tot,
                                                uint32_t* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = n_bins >= kT ? n_bins / kT : 1;           // bins per thread, walked from the top digit down
  const int n_act = n_bins / per;
  uint32_t local = 0;
  if (tid < n_act) {
    const int first = n_bins - (tid + 1) * per;              // the thread's bins are [first, first + per)
    if (per % 4 == 0) {                                      // 16-byte loads: consecutive threads, consecutive quads
      const uint4* q = reinterpret_cast<const uint4*>(hist + first);
      for (int j = 0; j < per / 4; ++j) { const uint4 v = q[j]; local += (v.x + v.y) + (v.z + v.w); }
    } else {
      for (int j = 0; j < per; ++j) local += hist[first + j];
    }
  }
  uint32_t incl = local;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) warp_tot[warp] = (int)incl;
  __syncthreads();
  uint32_t excl = incl - local;
  excl += (uint32_t)warps_before(warp_tot, warp, lane);
  if (tid < n_act && excl < k_rem && k_rem <= excl + local) {
    uint32_t acc = excl;
    for (int j = 0; j < per; ++j) {
      const int bin = n_bins - 1 - (tid * per + j);
      const uint32_t c = hist[bin];
      if (k_rem <= acc + c) {
        out[0] = (uint32_t)bin; out[1] = k_rem - acc; out[2] = c;
        break;
      }
      acc += c;
    }
  }
  __syncthreads();
}

// The block ranks the n <= min(kT, kRankList) candidates in sc.small, a thread each: returns the k_rem-th largest value,
// sets k_out to the rank left among the candidates equal to it and n_equal to their number.  A barrier lies between the
// list's last update and this call.
template <int kT>
__device__ __forceinline__ unsigned long long rank_select(Scratch& sc, int n, uint32_t k_rem, uint32_t& k_out, uint32_t& n_equal) {
  if ((int)threadIdx.x < n) {
    const unsigned long long v = sc.small[threadIdx.x];
    uint32_t gt = 0, ge = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const unsigned long long o = sc.small[j];
      gt += o > v;
      ge += o >= v;
    }
    if (gt < k_rem && k_rem <= ge) { sc.sel_x = v; sc.sel[1] = k_rem - gt; sc.sel[2] = ge - gt; }   // equal candidates agree
  }
  __syncthreads();
  k_out = sc.sel[1];
  n_equal = sc.sel[2];
  return sc.sel_x;
}

// One warp ranks at most 32 candidates held one per lane (lanes >= n hold nothing): returns the k_rem-th largest value in
// every lane.
__device__ __forceinline__ uint32_t warp_rank_select32(uint32_t v, int n, uint32_t k_rem, int lane) {
  uint32_t gt = 0, ge = 0;
  for (int j = 0; j < n; ++j) {
    const uint32_t o = __shfl_sync(kFull, v, j);
    gt += o > v;
    ge += o >= v;
  }
  const bool hit = lane < n && gt < k_rem && k_rem <= ge;
  const unsigned who = __ballot_sync(kFull, hit);
  return __shfl_sync(kFull, v, __ffs(who) - 1);
}

// Calls f(item, index) for items tid, tid + kT, .. of [0, n).  Items outside shared memory come eight loads at a time: they
// are read through L2, and f's atomics would hold every load back until the one before is used.
template <int kT, class Load, class F>
__device__ __forceinline__ void for_items(bool far, int n, Load&& load, F&& f) {
  if (!far) {
    for (int i = threadIdx.x; i < n; i += kT) f(load(i), i);
    return;
  }
  for (int i0 = threadIdx.x; i0 < n; i0 += 8 * kT) {
    decltype(load(0)) v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = load(min(i0 + j * kT, n - 1));
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (i0 + j * kT < n) f(v[j], i0 + j * kT);
  }
}

// Sets bit i of imp_mask for the k items with the largest keys[0..n); equal keys are admitted in ascending
// index order.  Exact.  The first round is a histogram of the keys' upper halves alone (32-bit arithmetic, warp-level
// minimum and maximum), over (upper half - smallest upper half) from the top bit in which they differ at all, so that the
// bins are spread whatever the keys' common magnitude; usually at most 256 keys are left in the bin of the k-th largest
// and are ranked directly (24 of them by one warp with 64-bit shuffles took 3 of the step's 10 thousand cycles).
// Otherwise radix rounds over the whole keys follow; then one ordered pass marks the members.  Called by all threads of the
// block; imp_mask must be zero on entry; 0 < k < n.
// copy: optional shared memory for n words; keys that are not in shared memory are then read whole only where it matters
// (the sweeps over 32768 keys took 9 thousand cycles each through L2).
template <int kT>
__device__ __forceinline__ void mark_top_keys(const unsigned long long* keys, int n, int k, uint32_t* imp_mask,
                                              Scratch& sc, uint32_t* copy = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  if (n <= 32) {                                       // one warp ranks every item: larger keys first, then lower index
    if (warp == 0) {
      const unsigned long long v = lane < n ? keys[lane] : 0ull;
      int before = 0;
      for (int j = 0; j < n; ++j) {
        const unsigned long long o = __shfl_sync(kFull, v, j);
        before += o > v || (o == v && j < lane);
      }
      const unsigned imp_b = __ballot_sync(kFull, lane < n && before < k);
      if (lane == 0) imp_mask[0] = imp_b;
    }
    __syncthreads();
    return;
  }
  int r_lo, r_hi;
  warp_range<kT>(n, warp, r_lo, r_hi);
  const bool far = !__isShared(keys), far_upper = far && !copy;
  const auto upper_word = [&](int i) { return reinterpret_cast<const uint32_t*>(keys)[2 * i + 1]; };
  const auto upper = [&](int i) { return copy ? copy[i] : upper_word(i); };
  const auto whole = [&](int i) { return keys[i]; };

  // smallest and largest upper half
  uint32_t lo32 = 0xFFFFFFFFu, hi32 = 0u;
  for_items<kT>(far, n, upper_word, [&](uint32_t x, int i) {
    lo32 = min(lo32, x);
    hi32 = max(hi32, x);
    if (copy) copy[i] = x;
  });
  lo32 = __reduce_min_sync(kFull, lo32);
  hi32 = __reduce_max_sync(kFull, hi32);
  if (lane == 0) sc.red[warp] = (unsigned long long)hi32 << 32 | lo32;
  for (int i = tid; i < kBins; i += kT) sc.hist[i] = 0;
  if (tid == 0) sc.small_n = 0;
  __syncthreads();
  {
    const unsigned long long v = sc.red[lane < kT / 32 ? lane : 0];
    lo32 = __reduce_min_sync(kFull, (uint32_t)v);
    hi32 = __reduce_max_sync(kFull, (uint32_t)(v >> 32));
  }
  const int bits = hi32 > lo32 ? 32 - __clz(hi32 - lo32) : 1, shift32 = bits > kDigitBits ? bits - kDigitBits : 0;
  for_items<kT>(far_upper, n, upper, [&](uint32_t x, int) { atomicAdd(&sc.hist[(x - lo32) >> shift32], 1u); });
  __syncthreads();
  find_digit_desc<kT>(sc.hist, kBins, (uint32_t)k, sc.warp_tot, sc.sel);
  const uint32_t digit = sc.sel[0], k_in_bin = sc.sel[1], live0 = sc.sel[2];

  unsigned long long kth;                              // the k-th largest key ..
  uint32_t k_rem, n_equal;                             // .. and how many of the n_equal keys equal to it are admitted
  constexpr uint32_t kDirect = kT < kRankList ? kT : kRankList;
  if (live0 <= kDirect) {
    for_items<kT>(far_upper, n, upper, [&](uint32_t x, int i) {
      if ((x - lo32) >> shift32 == digit) sc.small[atomicAdd(&sc.small_n, 1u)] = keys[i];
    });
    __syncthreads();
    kth = rank_select<kT>(sc, (int)live0, k_in_bin, k_rem, n_equal);
  } else {
    // radix rounds over x = key - base, base = the smallest upper half with zeros below: x has `rem` significant bits;
    // `top` is the value of the bits of x above them chosen so far.  The first digit is known.
    const unsigned long long base = (unsigned long long)lo32 << 32;
    int rem = 32 + shift32;
    unsigned long long top = digit;
    k_rem = k_in_bin;
    n_equal = live0;
    while (rem > 0) {
      const int w = rem < kDigitBits ? rem : kDigitBits, shift = rem - w, n_bins = 1 << w;
      __syncthreads();                                 // sc.sel and sc.hist are rewritten
      for (int i = tid; i < n_bins; i += kT) sc.hist[i] = 0;
      if (tid == 0) sc.small_n = 0;
      __syncthreads();
      for_items<kT>(far, n, whole, [&](unsigned long long key, int) {
        const unsigned long long x = key - base;
        if ((x >> rem) == top) atomicAdd(&sc.hist[(uint32_t)(x >> shift) & (uint32_t)(n_bins - 1)], 1u);
      });
      __syncthreads();
      find_digit_desc<kT>(sc.hist, n_bins, k_rem, sc.warp_tot, sc.sel);
      top = (top << w) | sc.sel[0];
      k_rem = sc.sel[1];
      const uint32_t live = sc.sel[2];
      n_equal = live;                                  // exact once no bits are left
      rem = shift;
      if (rem > 0 && live <= kDirect) {   // few candidates: ranked by their remaining bits
        for_items<kT>(far, n, whole, [&](unsigned long long key, int) {
          const unsigned long long x = key - base;
          if ((x >> rem) == top) sc.small[atomicAdd(&sc.small_n, 1u)] = x;
        });
        __syncthreads();
        uint32_t k_out;
        top = rank_select<kT>(sc, (int)live, k_rem, k_out, n_equal);
        k_rem = k_out;
        rem = 0;
      }
    }
    kth = base + top;
  }
  if (k_rem == n_equal && copy) {                      // no tie is cut (the usual case): everything >= kth is in
    const uint32_t kth_hi = (uint32_t)(kth >> 32);
    for (int base_i = r_lo; base_i < r_hi; base_i += 32) {
      const int i = base_i + lane;
      const uint32_t x = i < r_hi ? copy[i] : 0u;
      const unsigned imp_b = __ballot_sync(kFull, i < r_hi && (x > kth_hi || (x == kth_hi && keys[i] >= kth)));
      if (lane == 0) imp_mask[base_i >> 5] = imp_b;
    }
    __syncthreads();
    return;
  }
  if (k_rem == n_equal) {
    for (int base_i = r_lo; base_i < r_hi; base_i += 8 * 32) {
      unsigned long long key[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) key[j] = base_i + 32 * j + lane < r_hi ? keys[base_i + 32 * j + lane] : 0ull;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (base_i + 32 * j >= r_hi) break;
        const unsigned imp_b = __ballot_sync(kFull, base_i + 32 * j + lane < r_hi && key[j] >= kth);
        if (lane == 0) imp_mask[(base_i >> 5) + j] = imp_b;
      }
    }
    __syncthreads();
    return;
  }
  int n_eq = 0;
  for (int i = r_lo + lane; i < r_hi; i += 32) n_eq += (keys[i] == kth);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) n_eq += __shfl_xor_sync(kFull, n_eq, d);
  __syncthreads();                                     // warp_tot may still be read by the digit search
  if (lane == 0) sc.warp_tot[warp] = n_eq;
  __syncthreads();
  int eq_before = 0;
  eq_before += warps_before(sc.warp_tot, warp, lane);
  for (int base_i = r_lo; base_i < r_hi; base_i += 32) {
    const int i = base_i + lane;
    const unsigned long long key = i < r_hi ? keys[i] : 0ull;
    const bool eq = i < r_hi && key == kth;
    const unsigned eq_b = __ballot_sync(kFull, eq);
    const bool imp = i < r_hi && (key > kth || (eq && (uint32_t)(eq_before + __popc(eq_b & lt_mask)) < k_rem));
    const unsigned imp_b = __ballot_sync(kFull, imp);
    if (lane == 0) imp_mask[base_i >> 5] = imp_b;
    eq_before += __popc(eq_b);
  }
  __syncthreads();
}

// Writes the members of imp_mask | rep_mask in ascending order (kind: 1 for members of rep_mask), counted from item `first`.
// Called by all threads of the block after the masks are complete.
template <int kT>
__device__ __forceinline__ void emit_kept(const uint32_t* imp_mask, const uint32_t* rep_mask, int n_words,
                                          int32_t* out_idx, uint8_t* out_kind, Scratch& sc, int first = 0) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // every thread takes a contiguous run of mask BYTES (8 items each): with fewer words than threads a word-wise
  // split would leave most threads idle and the others with up to 32 serial stores
  const int n_bytes = 4 * n_words;
  const int bpt = (n_bytes + kT - 1) / kT;
  const int b_lo = min(n_bytes, tid * bpt), b_hi = min(n_bytes, b_lo + bpt);
  auto byte_of = [](const uint32_t* mask, int b) -> uint32_t { return (mask[b >> 2] >> (8 * (b & 3))) & 0xFFu; };
  int cnt = 0;
  for (int b = b_lo; b < b_hi; ++b) cnt += __popc(byte_of(imp_mask, b) | byte_of(rep_mask, b));
  int incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += v;
  }
  __syncthreads();                          // warp_tot may still be read by an earlier phase
  if (lane == 31) sc.warp_tot[warp] = incl;
  __syncthreads();
  int pos = incl - cnt;
  pos += warps_before(sc.warp_tot, warp, lane);
  for (int b = b_lo; b < b_hi; ++b) {
    const uint32_t rep = byte_of(rep_mask, b);
    uint32_t bits = byte_of(imp_mask, b) | rep;
    while (bits) {
      const int k = __ffs(bits) - 1;
      bits &= bits - 1;
      out_idx[pos] = first + 8 * b + k;
      if (out_kind) out_kind[pos] = (rep >> k) & 1u;
      ++pos;
    }
  }
}

}  // namespace sel
}  // namespace kvc

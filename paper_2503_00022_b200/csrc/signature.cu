// Stage 2: per-head thresholds and packed binary signatures (Algorithm 1 and Sec. 3.1 of the paper).
//
//   theta_select_kernel       theta = keep-th largest score of one (layer, sequence, head) row of up to 8192
//                             tokens: the row is read once into registers as order-preserving 32-bit keys, and
//                             the k-th largest is found by 12-bit radix histograms over (key - smallest key),
//                             starting at the top bit in which the row's keys differ at all; one warp ranks the
//                             last few candidates directly.  Usually one histogram pass.
//   theta_upper_kernel        the same result for rows of up to 32768 tokens, half of every key in shared memory.
//   theta_warp_kernel         the same search by one warp per row, for many short rows.
//   theta_stream_kernel       the same result for longer rows: MSB-first radix select (4 sweeps of 8 bits) that
//                             re-reads the row from memory (or from a shared-memory copy) in every sweep.
//   signature_pack_kernel     one block per (layer, 128 tokens): stages the [heads][tokens] tile of scores in shared
//                             memory with 16-byte row loads, then one thread per token compares its score of every
//                             head with that head's threshold and packs the bits; from the same tile it can add up
//                             the token's importance I(t) in float64, in the fixed order stage 3 defines, which
//                             saves stage 3 its own pass over the scores.
#include "select_common.cuh"

namespace kvc {

namespace {

constexpr int kSelectThreads = 512;
constexpr int kThetaBits = 12;                 // radix digit of theta_select_kernel
constexpr int kThetaBins = 1 << kThetaBits;

// float -> uint32 such that a < b  <=>  key(a) < key(b) (for non-NaN values)
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// kT threads, each holding up to kItems keys of the row: rows of up to kT * kItems tokens.  kMinB: resident blocks per
// SM the kernel is compiled for.  The kernel is a chain of short dependent steps, so what counts is how many rows an
// SM works on at once and how many threads share a row: measured for 1024 rows of 8192 scores, 512 threads x 16 keys
// at 4 blocks per SM (32 registers, a few spilled words) 16.2 us, 256 x 32 at 4 per SM 17.9 us, 512 x 16 at 2 per SM
// 20.3 us, 1024 x 8 at 2 per SM 19.7 us, 128 x 64 23.7 us.
template <int kT, int kItems, int kMinB>
__global__ void __launch_bounds__(kT, kMinB)
theta_select_kernel(Shape s, const float* __restrict__ scores, const int32_t* __restrict__ sig_keep,
                    float* __restrict__ theta) {
  __shared__ alignas(16) uint32_t hist[kThetaBins];
  __shared__ uint32_t red[2][32];
  __shared__ uint32_t small[sel::kSmallList];
  __shared__ uint32_t small_n;
  __shared__ uint32_t found[3];
  __shared__ int warp_tot[32];

  chain_wait();
  chain_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int h = blockIdx.x % s.Hq;
  const int seg = blockIdx.x / s.Hq;              // layer * n_seqs + seq
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int keep = __ldg(sig_keep + seg);
  float* out = theta + (size_t)seg * s.Hq + h;
  if (keep <= 0 || keep >= L) {
    if (tid == 0) *out = keep <= 0 ? __int_as_float(0x7F800000) : __int_as_float(0xFF800000);
    return;
  }
  const float* row = scores + ((size_t)layer * s.Hq + h) * s.T + t0;

  uint32_t key[kItems];
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = j * kT + tid;
    key[j] = i < L ? order_key(__ldg(row + i)) : 0u;
  }
#pragma unroll
  for (int j = 0; j < kItems; ++j)
    if (j * kT + tid < L) { lo = min(lo, key[j]); hi = max(hi, key[j]); }
  lo = __reduce_min_sync(sel::kFull, lo);
  hi = __reduce_max_sync(sel::kFull, hi);
  if (lane == 0) { red[0][warp] = lo; red[1][warp] = hi; }
  for (int i = tid; i < kThetaBins; i += kT) hist[i] = 0;
  if (tid == 0) small_n = 0;
  __syncthreads();
  lo = __reduce_min_sync(sel::kFull, lane < kT / 32 ? red[0][lane] : 0xFFFFFFFFu);
  hi = __reduce_max_sync(sel::kFull, lane < kT / 32 ? red[1][lane] : 0u);
  const uint32_t base = lo, range = hi - lo;
  // From here on key[j] holds x = key - base; slots past the end of the row hold 0, the row's minimum: they add to
  // the count of the lowest values only, which a rank counted from the top (keep < L) never reaches beyond the
  // real minimum itself.
#pragma unroll
  for (int j = 0; j < kItems; ++j) key[j] = j * kT + tid < L ? key[j] - base : 0u;

  // x has `rem` significant bits; `top` is the value of the bits of x above them chosen so far
  int rem = range ? 32 - __clz(range) : 0;
  uint32_t top = 0, k_rem = (uint32_t)keep;
  bool first = true;
  while (rem > 0) {
    const int w = rem < kThetaBits ? rem : kThetaBits, shift = rem - w, n_bins = 1 << w;
    if (first) {                                             // every x counts and has no bits above the digit
#pragma unroll
      for (int j = 0; j < kItems; ++j) atomicAdd(&hist[key[j] >> shift], 1u);
    } else {
      for (int i = tid; i < n_bins; i += kT) hist[i] = 0;
      if (tid == 0) small_n = 0;
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kItems; ++j)
        if (((key[j] >> 1) >> (rem - 1)) == top) atomicAdd(&hist[(key[j] >> shift) & (uint32_t)(n_bins - 1)], 1u);
    }
    first = false;
    __syncthreads();
    sel::find_digit_desc<kT>(hist, n_bins, k_rem, warp_tot, found);
    top = (top << w) | found[0];
    k_rem = found[1];
    const uint32_t live = found[2];
    rem = shift;
    if (rem > 0 && live <= (uint32_t)sel::kSmallList) {     // few candidates: one warp ranks them and finishes
#pragma unroll
      for (int j = 0; j < kItems; ++j)
        if ((key[j] >> rem) == top) small[atomicAdd(&small_n, 1u)] = key[j];
      __syncthreads();
      if (warp == 0) {
        const uint32_t x = sel::warp_rank_select32(lane < (int)live ? small[lane] : 0u, (int)live, k_rem, lane);
        if (lane == 0) *out = key_to_float(base + x);
      }
      return;
    }
    __syncthreads();                                         // hist and found are rewritten by the next step
  }
  if (tid == 0) *out = key_to_float(base + top);
}

// Rows of 8193 to 32768 tokens.  A row of full keys takes half of an SM's registers, so that one block an SM loaded,
// counted and searched in turn.  Here the upper halves of the keys go to shared memory, which lets two blocks of 1024
// threads share an SM: one loads while the other counts.  The first histogram covers the upper halves (128 bins an
// octave); the keys in the bin of the k-th largest are read again and ranked a thread each.  1024 rows of 32768 scores:
// 92 -> 62 us (the signature stage 127 -> 98).
constexpr int kListKeys = 1024;

__global__ void __launch_bounds__(1024, 2)
theta_upper_kernel(Shape s, const float* __restrict__ scores, const int32_t* __restrict__ sig_keep, float* __restrict__ theta) {
  constexpr int kT = 1024;
  extern __shared__ __align__(16) uint16_t upper[];   // [max_seqlen], read in pairs
  __shared__ alignas(16) uint32_t hist[kThetaBins];
  __shared__ uint32_t list[kListKeys];
  __shared__ uint32_t red[32], list_n, found[3];
  __shared__ int warp_tot[32];
  chain_wait();
  chain_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int h = blockIdx.x % s.Hq;
  const int seg = blockIdx.x / s.Hq;              // layer * n_seqs + seq
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int keep = __ldg(sig_keep + seg);
  float* out = theta + (size_t)seg * s.Hq + h;
  if (keep <= 0 || keep >= L) {
    if (tid == 0) *out = keep <= 0 ? __int_as_float(0x7F800000) : __int_as_float(0xFF800000);
    return;
  }
  const float* row = scores + ((size_t)layer * s.Hq + h) * s.T + t0;

  uint32_t lo = 0xFFFFu, hi = 0u;
  for (int i0 = tid; i0 < L; i0 += 8 * kT) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __ldg(row + min(i0 + j * kT, L - 1));
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t x = order_key(v[j]) >> 16;
      lo = min(lo, x);
      hi = max(hi, x);
      if (i0 + j * kT < L) upper[i0 + j * kT] = (uint16_t)x;
    }
  }
  for (int i = tid; i < kThetaBins; i += kT) hist[i] = 0;
  if (tid == 0) list_n = 0;
  // f(upper half, token), two neighbouring tokens a thread
  auto each = [&](auto&& f) {
    const uint32_t* pairs = reinterpret_cast<const uint32_t*>(upper);
    for (int p = tid; 2 * p < L; p += kT) {
      const uint32_t x = pairs[p];
      f(x & 0xFFFFu, 2 * p);
      if (2 * p + 1 < L) f(x >> 16, 2 * p + 1);
    }
  };
  lo = __reduce_min_sync(sel::kFull, lo);
  hi = __reduce_max_sync(sel::kFull, hi);
  if (lane == 0) red[warp] = hi << 16 | lo;
  __syncthreads();
  lo = __reduce_min_sync(sel::kFull, red[lane] & 0xFFFFu);
  hi = __reduce_max_sync(sel::kFull, red[lane] >> 16);
  const int bits = hi > lo ? 32 - __clz(hi - lo) : 0, shift = bits > kThetaBits ? bits - kThetaBits : 0;
  each([&](uint32_t x, int) { atomicAdd(&hist[(x - lo) >> shift], 1u); });
  __syncthreads();
  sel::find_digit_desc<kT>(hist, kThetaBins, (uint32_t)keep, warp_tot, found);
  const uint32_t digit = found[0], live = found[2];
  uint32_t k_rem = found[1];
  if (live <= (uint32_t)kListKeys) {
    each([&](uint32_t x, int i) {
      if ((x - lo) >> shift == digit) list[atomicAdd(&list_n, 1u)] = order_key(__ldg(row + i));
    });
    __syncthreads();
    if (tid < (int)live) {
      const uint32_t v = list[tid];
      uint32_t gt = 0, ge = 0;
#pragma unroll 4
      for (int j = 0; j < (int)live; ++j) {
        const uint32_t o = list[j];
        gt += o > v;
        ge += o >= v;
      }
      if (gt < k_rem && k_rem <= ge) *out = key_to_float(v);       // equal keys agree
    }
    return;
  }
  // more than that in one bin (ties): radix rounds over the whole keys, read again in every round
  const uint32_t base = lo << 16;
  int rem = 16 + shift;                                      // bits of key - base below the ones in top
  uint32_t top = digit;
  while (rem > 0) {
    const int w = rem < kThetaBits ? rem : kThetaBits, sh = rem - w, n_bins = 1 << w;
    __syncthreads();
    for (int i = tid; i < n_bins; i += kT) hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < L; i += kT) {
      const uint32_t x = order_key(__ldg(row + i)) - base;
      if (x >> rem == top) atomicAdd(&hist[(x >> sh) & (uint32_t)(n_bins - 1)], 1u);
    }
    __syncthreads();
    sel::find_digit_desc<kT>(hist, n_bins, k_rem, warp_tot, found);
    top = top << w | found[0];
    k_rem = found[1];
    rem = sh;
  }
  if (tid == 0) *out = key_to_float(base + top);
}

// One warp per row, for rows of up to 32 * kItems tokens: the same search as theta_select_kernel without a block's
// barriers, and with as many rows in flight as an SM has warps.  Short rows come in large numbers (a serving batch of 16
// sequences x 32 layers x 32 heads of 736 tokens is 16384 rows), where a block per row spends its time in barriers: the
// signature stage took 99 us with it and takes 62 us with this kernel.
constexpr int kRowWarps = 8;
constexpr int kRowBits = 9;
constexpr int kRowBins = 1 << kRowBits;

template <int kItems>
__global__ void __launch_bounds__(kRowWarps * 32, kItems == 32 ? 3 : 4)
theta_warp_kernel(Shape s, const float* __restrict__ scores, const int32_t* __restrict__ sig_keep,
                  float* __restrict__ theta, unsigned n_rows) {
  __shared__ alignas(16) uint32_t hist_sh[kRowWarps][kRowBins];
  __shared__ uint32_t small_sh[kRowWarps][sel::kSmallList];
  __shared__ uint32_t small_n_sh[kRowWarps];
  chain_wait();
  chain_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned r = blockIdx.x * kRowWarps + warp;
  if (r >= n_rows) return;
  uint32_t* hist = hist_sh[warp];
  const int h = r % s.Hq;
  const int seg = r / s.Hq;                       // layer * n_seqs + seq
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int keep = __ldg(sig_keep + seg);
  if (keep <= 0 || keep >= L) {
    if (lane == 0) theta[r] = keep <= 0 ? __int_as_float(0x7F800000) : __int_as_float(0xFF800000);
    return;
  }
  const float* row = scores + ((size_t)layer * s.Hq + h) * s.T + t0;
  uint32_t key[kItems];
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int j = 0; j < kItems; ++j) key[j] = j * 32 + lane < L ? order_key(__ldg(row + j * 32 + lane)) : 0u;
#pragma unroll
  for (int j = 0; j < kItems; ++j)
    if (j * 32 + lane < L) { lo = min(lo, key[j]); hi = max(hi, key[j]); }
  const uint32_t base = __reduce_min_sync(sel::kFull, lo), range = __reduce_max_sync(sel::kFull, hi) - base;
#pragma unroll
  for (int j = 0; j < kItems; ++j) key[j] -= base;            // slots past the end of the row are left out below

  int rem = range ? 32 - __clz(range) : 0;
  uint32_t top = 0, k_rem = (uint32_t)keep;
  while (rem > 0) {
    const int w = rem < kRowBits ? rem : kRowBits, shift = rem - w;
    uint4* h4 = reinterpret_cast<uint4*>(hist);
#pragma unroll
    for (int i = 0; i < kRowBins / 128; ++i) h4[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    if (lane == 0) small_n_sh[warp] = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kItems; ++j)
      if (j * 32 + lane < L && ((key[j] >> 1) >> (rem - 1)) == top) atomicAdd(&hist[(key[j] >> shift) & ((1u << w) - 1u)], 1u);
    __syncwarp();
    // lane l owns the kRowBins / 32 bins from kRowBins - 1 - l * 16 downwards (bins above the digit's width are empty)
    uint32_t c[kRowBins / 32], local = 0;
#pragma unroll
    for (int i = 0; i < kRowBins / 128; ++i) {
      const uint4 v = h4[(31 - lane) * (kRowBins / 128) + (kRowBins / 128 - 1 - i)];
      c[4 * i] = v.w; c[4 * i + 1] = v.z; c[4 * i + 2] = v.y; c[4 * i + 3] = v.x;
      local += (v.x + v.y) + (v.z + v.w);
    }
    uint32_t incl = local;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(sel::kFull, incl, d);
      if (lane >= d) incl += v;
    }
    uint32_t acc = incl - local, bin = 0, left = 0, live = 0;
    const bool mine = acc < k_rem && k_rem <= incl;
    if (mine) {
      bool found = false;
#pragma unroll
      for (int i = 0; i < kRowBins / 32; ++i) {
        if (!found && k_rem <= acc + c[i]) {
          found = true;
          bin = kRowBins - 1 - lane * (kRowBins / 32) - i; left = k_rem - acc; live = c[i];
        }
        acc += c[i];
      }
    }
    const int src = __ffs(__ballot_sync(sel::kFull, mine)) - 1;
    top = (top << w) | __shfl_sync(sel::kFull, bin, src);
    k_rem = __shfl_sync(sel::kFull, left, src);
    live = __shfl_sync(sel::kFull, live, src);
    rem = shift;
    if (rem > 0 && live <= (uint32_t)sel::kSmallList) {      // few candidates: ranked directly
#pragma unroll
      for (int j = 0; j < kItems; ++j)
        if (j * 32 + lane < L && (key[j] >> rem) == top) small_sh[warp][atomicAdd(&small_n_sh[warp], 1u)] = key[j];
      __syncwarp();
      top = sel::warp_rank_select32(lane < (int)live ? small_sh[warp][lane] : 0u, (int)live, k_rem, lane);
      rem = 0;
    }
  }
  if (lane == 0) theta[r] = key_to_float(base + top);
}

__global__ void __launch_bounds__(kSelectThreads)
theta_stream_kernel(Shape s, const float* __restrict__ scores, const int32_t* __restrict__ sig_keep,
                    float* __restrict__ theta, int stage_row) {
  extern __shared__ uint32_t row_keys[];          // the row's order keys when it fits (stage_row), else unused
  __shared__ uint32_t hist[256];
  __shared__ uint32_t sel_prefix, sel_k;
  chain_wait();
  chain_trigger();

  const int h = blockIdx.x % s.Hq;
  const int seg = blockIdx.x / s.Hq;              // layer * n_seqs + seq
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int keep = __ldg(sig_keep + seg);
  float* out = theta + (size_t)seg * s.Hq + h;
  if (keep <= 0 || keep >= L) {
    if (threadIdx.x == 0) *out = keep <= 0 ? __int_as_float(0x7F800000) : __int_as_float(0xFF800000);
    return;
  }
  const float* row = scores + ((size_t)layer * s.Hq + h) * s.T + t0;
  const int lane = threadIdx.x & 31;

  // When the row fits, its order keys are first copied into shared memory with independent, coalesced loads
  // (the sweeps below interleave every load with warp votes and atomics, which would expose the full global
  // latency once per element).
  if (stage_row) {
#pragma unroll 4
    for (int i = threadIdx.x; i < L; i += kSelectThreads) row_keys[i] = order_key(__ldg(row + i));
    __syncthreads();
  }

  uint32_t prefix = 0;       // selected high digits so far
  uint32_t k_rem = keep;     // rank among the elements that share the prefix
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 256; i += kSelectThreads) hist[i] = 0;
    __syncthreads();
    const uint32_t hi_mask = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
    for (int base = 0; base < L; base += kSelectThreads) {
      const int i = base + threadIdx.x;
      const bool in = i < L;
      const uint32_t key = !in ? 0u : stage_row ? row_keys[i] : order_key(__ldg(row + i));
      const bool live = in && ((key & hi_mask) == prefix);
      const uint32_t digit = (key >> shift) & 0xFFu;
      // high digits (sign, exponent) are the same for almost every score: one add per warp then;
      // low digits are spread over the 256 bins, where plain shared-memory atomics do not collide much
      const unsigned voters = __ballot_sync(0xFFFFFFFFu, live);
      if (voters) {
        const uint32_t d0 = __shfl_sync(0xFFFFFFFFu, digit, __ffs(voters) - 1);
        if (__all_sync(0xFFFFFFFFu, !live || digit == d0)) {
          if (lane == 0) atomicAdd(&hist[d0], __popc(voters));
        } else if (live) {
          atomicAdd(&hist[digit], 1u);
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      // lane l owns the 8 bins 255-8l .. 248-8l (descending order of value)
      uint32_t local = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) local += hist[255 - 8 * lane - j];
      uint32_t incl = local;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += v;
      }
      const uint32_t excl = incl - local;
      if (excl < k_rem && k_rem <= incl) {
        uint32_t acc = excl;
        for (int j = 0; j < 8; ++j) {
          const uint32_t c = hist[255 - 8 * lane - j];
          if (k_rem <= acc + c) {
            sel_prefix = prefix | ((uint32_t)(255 - 8 * lane - j) << shift);
            sel_k = k_rem - acc;
            break;
          }
          acc += c;
        }
      }
    }
    __syncthreads();
    prefix = sel_prefix;
    k_rem = sel_k;
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = key_to_float(prefix);
}

// kImportance: also write I(t) = sum of the token's per-head scores (float64; heads ascending inside each KV
// group, then the group sums ascending: sequential IEEE additions, so the value is bit-reproducible).
// Grid: (token blocks, layers); a block owns kPackTok consecutive tokens of one layer.  Its [heads][tokens] tile of
// scores goes through shared memory: the loads are 16-byte, row-contiguous and all in flight at once (eight per
// thread at 32 heads), and the per-token walk over the heads afterwards reads shared memory without conflicts.
// Behind the thresholds' kernel it loads its scores before it waits for it: signature stage of 32 x 32 rows of 1001 tokens 17.2 ->
// 14.5 us, of 8 x 32 rows of 8192 16.1 -> 14.9, of 16 x 32 x 32 rows of 736 44.7 -> 43.8.  (A thread that holds its token's 32
// scores in registers instead of the staged tile: 5 to 10 % slower for 8 heads and for large grids.)
// The thresholds of the block's sequence sit in shared memory when all its tokens belong to one sequence (always,
// with one sequence per batch); else every thread reads its own sequence's row.
constexpr int kPackTok = 128;
#ifndef KVC_PACK_MINB
#define KVC_PACK_MINB 8                 // resident blocks per SM the pack kernel is compiled for (registers per thread)
#endif

template <bool kImportance>
__global__ void __launch_bounds__(kPackTok, KVC_PACK_MINB)
signature_pack_kernel(Shape s, const float* __restrict__ scores, const float* __restrict__ theta,
                      uint32_t* __restrict__ sigs, double* __restrict__ importance, int vec_ok, int early) {
  extern __shared__ float4 tile4[];                   // [Hq][kPackTok] float
  float* tile = reinterpret_cast<float*>(tile4);
  __shared__ float th_sh[128];
  if (!early) chain_wait();                       // early: the thresholds' kernel is the launch before, the scores are older
  const int layer = blockIdx.y;
  const int tok0 = blockIdx.x * kPackTok, tok = tok0 + threadIdx.x;
  const int n_tok = min(kPackTok, s.T - tok0);
  const float* base = scores + (size_t)layer * s.Hq * s.T + tok0;
  if (vec_ok && n_tok == kPackTok) {                  // rows start on 16-byte boundaries
#pragma unroll 8
    for (int i = threadIdx.x; i < s.Hq * (kPackTok / 4); i += kPackTok) {
      const int h = i / (kPackTok / 4), c = i % (kPackTok / 4);
      tile4[i] = __ldcg(reinterpret_cast<const float4*>(base + (size_t)h * s.T) + c);
    }
  } else {
#pragma unroll 8
    for (int h = 0; h < s.Hq; ++h)
      tile[h * kPackTok + threadIdx.x] = (int)threadIdx.x < n_tok ? __ldcg(base + (size_t)h * s.T + threadIdx.x) : 0.f;
  }
  const int seq0 = seq_of_token(s.cu_seqlens, s.n_seqs, tok0);
  if (early) chain_wait();
  chain_trigger();
  const bool one_seq = tok0 + n_tok <= __ldg(s.cu_seqlens + seq0 + 1);
  if (one_seq)
    for (int h = threadIdx.x; h < s.Hq; h += kPackTok) th_sh[h] = __ldcg(theta + ((size_t)layer * s.n_seqs + seq0) * s.Hq + h);
  __syncthreads();
  if ((int)threadIdx.x >= n_tok) return;
  const float* th = one_seq ? th_sh
                            : theta + ((size_t)layer * s.n_seqs + seq_of_token(s.cu_seqlens, s.n_seqs, tok)) * s.Hq;
  const float* col = tile + threadIdx.x;
  uint32_t* out = sigs + ((size_t)layer * s.T + tok) * s.W;
  double total = 0.0, group = 0.0;
  int in_group = 0;
  for (int w = 0; w < s.W; ++w) {
    uint32_t word = 0;
    const int nb = min(32, s.Hq - 32 * w);
#pragma unroll 8
    for (int b = 0; b < nb; ++b) {
      const float v = col[(32 * w + b) * kPackTok];
      word |= (uint32_t)(v >= th[32 * w + b]) << b;
      if constexpr (kImportance) {
        group = __dadd_rn(group, (double)v);
        if (++in_group == s.G) { total = __dadd_rn(total, group); group = 0.0; in_group = 0; }
      }
    }
    out[w] = word;
  }
  if constexpr (kImportance) importance[(size_t)layer * s.T + tok] = __dadd_rn(total, 0.0);       // -0.0 -> +0.0
}

}  // namespace

int launch_signature(const Shape& s, const float* scores, const int32_t* sig_keep, const float* theta_in,
                     uint32_t* sigs, float* theta, double* importance, cudaStream_t stream) {
  if (s.T == 0) return KVCRUSH_OK;
  const float* th = theta_in;
  if (!theta_in) {
    const unsigned blocks = (unsigned)s.n_layers * s.n_seqs * s.Hq;
    const int m = s.max_seqlen;
    // A warp per row up to 512 tokens (stage at 1024 rows of 400 tokens: 11.8 -> 7.5 us); up to 1024 tokens only for
    // more rows than the chip holds as blocks (8 an SM): its chain over 32 keys a lane is longer than the block's
    // (32 rows of 1001 tokens: 8.9 against 7.3 us).
    const unsigned warp_blocks = (blocks + kRowWarps - 1) / kRowWarps;
    auto by_warp = [&](auto kern) {
      return launch_chained(kern, dim3(warp_blocks), dim3(kRowWarps * 32), 0, stream, 1, s, scores, sig_keep, theta, blocks);
    };
    auto by_block = [&](auto kern, int threads) {
      return launch_chained(kern, dim3(blocks), dim3(threads), 0, stream, 1, s, scores, sig_keep, theta);
    };
    int rc;
    if (m <= 256) rc = by_warp(theta_warp_kernel<8>);
    else if (m <= 512) rc = by_warp(theta_warp_kernel<16>);
    else if (m <= 1024 && blocks > 8u * (unsigned)sm_count()) rc = by_warp(theta_warp_kernel<32>);
    else if (m <= 2048) rc = by_block(theta_select_kernel<256, 8, 8>, 256);
    else if (m <= 4096) rc = by_block(theta_select_kernel<512, 8, 4>, 512);
    else if (m <= 8192) rc = by_block(theta_select_kernel<512, 16, 4>, 512);
    else if (m <= 32768) {
      const size_t dyn = ((size_t)m * sizeof(uint16_t) + 15) / 16 * 16;
      if (allow_dynamic_smem(theta_upper_kernel, 32768 * (int)sizeof(uint16_t)) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
      rc = launch_chained(theta_upper_kernel, dim3(blocks), dim3(1024), dyn, stream, 1, s, scores, sig_keep, theta);
    }
    else {
      const size_t row_bytes = (size_t)m * sizeof(uint32_t);
      constexpr int kMaxRow = 200 * 1024;
      const int stage_row = row_bytes <= kMaxRow;
      const size_t dyn = stage_row ? row_bytes : 0;
      if (stage_row && allow_dynamic_smem(theta_stream_kernel, kMaxRow) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
      rc = launch_chained(theta_stream_kernel, dim3(blocks), dim3(kSelectThreads), dyn, stream, 1, s, scores, sig_keep, theta, stage_row);
    }
    if (rc != KVCRUSH_OK) return rc;
    th = theta;
  }
  const dim3 grid((unsigned)((s.T + kPackTok - 1) / kPackTok), (unsigned)s.n_layers);
  const size_t dyn = (size_t)s.Hq * kPackTok * sizeof(float);
  // 16-byte loads need every (layer, head) row to start on a 16-byte boundary
  const int vec_ok = s.T % 4 == 0 && reinterpret_cast<uintptr_t>(scores) % 16 == 0;
  auto kern = importance ? signature_pack_kernel<true> : signature_pack_kernel<false>;
  if (dyn > 40 * 1024 && allow_dynamic_smem(kern, 128 * kPackTok * (int)sizeof(float)) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
  return launch_chained(kern, grid, dim3(kPackTok), dyn, stream, 1, s, scores, th, sigs, importance, vec_ok, !theta_in);
}

// ---------------------------------------------------------------------------------------------------
// kvcrush_signature_static: the same two kernels, thresholds kept in library-owned device memory.
// ---------------------------------------------------------------------------------------------------
namespace {

// Thresholds of one call, [n_layers][n_seqs][n_q_heads].  Lives in the library image on every device.
static __device__ __align__(256) float g_static_theta[KVCRUSH_STATIC_THETA_MAX];

constexpr int kMaxDevices = 64;

// Device address of g_static_theta on the current device.  In host code the symbol's name is only a
// handle; the address a kernel can use comes from cudaGetSymbolAddress, looked up once per device.
int static_theta_ptr(float** out) {
  static float* cached[kMaxDevices] = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return KVCRUSH_ERR_CUDA;
  float* p = __atomic_load_n(&cached[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_static_theta) != cudaSuccess || !addr) return KVCRUSH_ERR_CUDA;
    p = static_cast<float*>(addr);
    __atomic_store_n(&cached[dev], p, __ATOMIC_RELEASE);
  }
  *out = p;
  return KVCRUSH_OK;
}

}  // namespace
}  // namespace kvc

extern "C" int kvcrush_signature_static(const kvcrush_problem_t* problem, const float* scores_dev,
                                        const int32_t* sig_keep_dev, uint32_t* sigs_dev,
                                        int32_t* status_dev, void* stream) {
  kvc::Shape s;
  const int rc = kvc::shape_from_problem(problem, &s);
  if (rc != KVCRUSH_OK) return rc;
  if (!scores_dev || !sig_keep_dev || !sigs_dev || !status_dev) return KVCRUSH_ERR_INVALID_ARG;
  if ((long long)s.n_layers * s.n_seqs * s.Hq > KVCRUSH_STATIC_THETA_MAX) return KVCRUSH_ERR_STATIC_LIMIT;
  float* theta = nullptr;
  const int prc = kvc::static_theta_ptr(&theta);
  if (prc != KVCRUSH_OK) return prc;
  return kvc::launch_signature(s, scores_dev, sig_keep_dev, nullptr, sigs_dev, theta, nullptr,
                               static_cast<cudaStream_t>(stream));
}

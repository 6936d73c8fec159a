// Stage 3: the kept set of every (layer, sequence) segment (Sec. 3 and Algorithm 2 of the paper).
//
//   importance_kernel      I(t) = sum of the per-head scores of token t (H2O's cumulative attention),
//                          float64, heads added in ascending order inside each KV group and the
//                          group sums added in ascending order; stored as an order-preserving
//                          64-bit key.  One thread per (layer, token), coalesced per-head rows.
//                          Skipped when the caller hands over I(t) (the signature stage can write it
//                          from the loads it does anyway).
//   select_segment_kernel  one CTA per segment:
//                            1. exact radix select of the B_imp-th largest key, ties admitted in
//                               ascending token order                         -> important set
//                            2. anchor; d_t = popc(sig_t xor anchor) for the other tokens
//                            3. stable counting sort by (d_t, t): every warp owns a contiguous
//                               token range, per-warp histograms, one scan, ordered scatter
//                            4. equal-frequency buckets of the sorted order; per bucket the member
//                               minimising  sum_{h: bit set} (m - 2 n_h)  (= L1 distance to the
//                               per-bit mean, up to a constant), ties to the lower token
//                            5. kept = important U representatives, ascending token index
// A chain of short block-wide steps in one CTA per segment, bound by their latencies (8192 tokens, thousand cycles: staging
// 4.7, top-k 6.8, sort 7.7, buckets 13 to 21, output 2.9; device time 20.5 -> 18.4 us for 32 such segments, 10.1 -> 8.2 us
// for one of 1001 tokens); from about 13000 tokens on by instructions and L2 reads (32 segments of 32768 tokens 117 -> 69 us).
// Few segments of 8192 tokens or more take select_cluster_kernel, four or eight blocks a segment: 32 of 32768 tokens, with the
// keys' conversion, 71 -> 34 us.
// All decisions are integer or exact float64 comparisons, so the result is unique.
#include <atomic>
#include <type_traits>

#include "select_common.cuh"

namespace kvc {

namespace {

using sel::kFull;
using sel::head_mask;
constexpr int kMaxBins = 129;              // Hamming distances 0..128

// Order-preserving 64-bit key of a float64 importance; tokens kept by decree (the first keep_initial and the last
// keep_recent of a sequence of L tokens) rank as +infinity.
__device__ __forceinline__ unsigned long long importance_key(double v, int t, int L, int keep_initial, int keep_recent) {
  if (t < keep_initial || t >= L - keep_recent) v = __longlong_as_double(0x7FF0000000000000LL);
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__global__ void __launch_bounds__(256)
importance_kernel(Shape s, const float* __restrict__ scores, int keep_initial, int keep_recent,
                  unsigned long long* __restrict__ keys) {
  chain_wait();
  chain_trigger();
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long long)s.n_layers * s.T) return;
  const int layer = (int)(gid / s.T), tok = (int)(gid - (long long)layer * s.T);
  const float* sc = scores + (size_t)layer * s.Hq * s.T + tok;
  // the additions are sequential by definition (fixed order = bit-reproducible ranking); the loads are not,
  // so they are issued eight at a time ahead of the adds that consume them
  double total = 0.0, group = 0.0;
  int in_group = 0;
  for (int h0 = 0; h0 < s.Hq; h0 += 8) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = h0 + j < s.Hq ? __ldg(sc + (size_t)(h0 + j) * s.T) : 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (h0 + j < s.Hq) {
        group = __dadd_rn(group, (double)v[j]);
        if (++in_group == s.G) { total = __dadd_rn(total, group); group = 0.0; in_group = 0; }
      }
    }
  }
  total = __dadd_rn(total, 0.0);           // -0.0 -> +0.0
  int t = 0, L = 0x7FFFFFFF;
  if (keep_recent > 0 || keep_initial > 0) {   // the first / last tokens of a sequence are important by decree
    const int seq = seq_of_token(s.cu_seqlens, s.n_seqs, tok);
    t = tok - __ldg(s.cu_seqlens + seq);
    L = __ldg(s.cu_seqlens + seq + 1) - __ldg(s.cu_seqlens + seq);
  }
  keys[gid] = importance_key(total, t, L, keep_initial, keep_recent);
}

// Keys from an importance array the caller supplies (segments too long for the shared-memory copy, where the
// conversion happens otherwise).
__global__ void __launch_bounds__(256)
importance_keys_kernel(Shape s, const double* __restrict__ imp, int keep_initial, int keep_recent,
                       unsigned long long* __restrict__ keys) {
  chain_wait();
  chain_trigger();
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long long)s.n_layers * s.T) return;
  const int tok = (int)(gid % s.T);
  const int seq = seq_of_token(s.cu_seqlens, s.n_seqs, tok);
  const int t0 = __ldg(s.cu_seqlens + seq);
  keys[gid] = importance_key(imp[gid], tok - t0, __ldg(s.cu_seqlens + seq + 1) - t0, keep_initial, keep_recent);
}

// sum over the GW lanes of the group that starts at lane g0: popc(mine & theirs); lanes without a member hold zeros
template <int W, int GW>
__device__ __forceinline__ int group_and_popc(const uint32_t (&mine)[4], int g0) {
  int common = 0;
#pragma unroll
  for (int u = 0; u < GW; ++u)
#pragma unroll
    for (int w = 0; w < W; ++w) common += __popc(mine[w] & __shfl_sync(kFull, mine[w], g0 + u));
  return common;
}

struct SelectArgs {
  const unsigned long long* keys;     // [n_layers][T] importance keys; or, when NULL,
  const double* imp;                  // [n_layers][T] importance values, turned into keys while they are staged
  int keep_initial, keep_recent;      // tokens important by decree (applied with imp; keys have them built in)
  const uint32_t* sigs;               // [n_layers][T][W]
  const int32_t* budget_imp;
  const int32_t* budget_rep;
  int anchor_mode;
  const uint32_t* anchor_bits;
  int anchor_per_segment;
  const int32_t* cu_kept;
  int32_t* idx;
  uint8_t* kind;
  int32_t* n_kept;                    // optional [n_layers][n_seqs]: tokens kept per segment
  int32_t* sorted;                    // [n_layers][T] scratch: grouped tokens in (d, t) order (segments not staged)
  int mask_words;                     // words of one membership mask in shared memory
  int stage_words;                    // max_seqlen rounded up to a multiple of 4 (one staged int32 per token)
  int stage_sig, stage_sorted;        // kLong: which of the two live in shared memory (sorted: as 16-bit indices)
};

// W: signature words per token (compile time: the per-word loops unroll).
// kLong: segments whose keys, signatures and sorted order do not all fit in shared memory.  Of those the signatures come
// first, which the bucket step gathers one by one, then the sorted order as 16-bit indices; the keys' upper halves are
// copied into the signatures' place while the top k are looked for.
template <int W, bool kLong, int kT>
__global__ void __launch_bounds__(kT, 1024 / kT)
select_segment_kernel(Shape s, SelectArgs a) {
  constexpr int kWarps = kT / 32;
  extern __shared__ __align__(16) uint32_t dyn_smem[];
  uint32_t* imp_mask = dyn_smem;
  uint32_t* rep_mask = dyn_smem + a.mask_words;

  // the scratch of the top-k step and the per-warp histograms of the sort are not in use at the same time
  __shared__ union { sel::Scratch sc; int warp_hist[kWarps][kMaxBins]; } shared;
  sel::Scratch& sc = shared.sc;
  int (&warp_hist)[kWarps][kMaxBins] = shared.warp_hist;
  __shared__ int bin_base[kMaxBins + 1];
  __shared__ int bit_cnt[128];
  __shared__ uint32_t anchor_sh[4];
  chain_wait();
  chain_trigger();

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int seg = blockIdx.x;
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int b_imp = max(0, __ldg(a.budget_imp + seg));
  const int b_rep = max(0, __ldg(a.budget_rep + seg));
  int32_t* out_idx = a.idx + __ldg(a.cu_kept + seg);
  uint8_t* out_kind = a.kind ? a.kind + __ldg(a.cu_kept + seg) : nullptr;

  if (a.n_kept && tid == 0) a.n_kept[seg] = (int)min((long long)b_imp + b_rep, (long long)L);
  if ((long long)b_imp + b_rep >= L) {             // budget covers the sequence: keep everything
    for (int i = tid; i < L; i += kT) {
      out_idx[i] = i;
      if (out_kind) out_kind[i] = 0;
    }
    return;
  }

  // The segment's arrays are read many times with dependent addresses (radix sweeps, counting-sort sweeps, one gather
  // per bucket), so whatever fits is first copied into shared memory; the rest is read through L2.  The pointers below
  // are generic and point to either place.
  const unsigned long long* keys = a.keys ? a.keys + (size_t)layer * s.T + t0 : nullptr;
  const uint32_t* sig = a.sigs + ((size_t)layer * s.T + t0) * W;
  uint32_t* arena = dyn_smem + 2 * a.mask_words;
  uint32_t* sig_sh = kLong && !a.stage_sig ? nullptr : arena;
  if (sig_sh) arena += a.stage_words * W;
  int32_t* sorted = kLong ? a.sorted + (size_t)layer * s.T + t0 : reinterpret_cast<int32_t*>(arena);
  uint16_t* sorted16 = kLong && a.stage_sorted ? reinterpret_cast<uint16_t*>(arena) : nullptr;
  arena += a.stage_words;
  uint32_t* sort_code = arena;           // !kLong, per token: distance | position among the warp's tokens of that distance << 8
  auto sorted_at = [&](int i) { return kLong && sorted16 ? (int)sorted16[i] : sorted[i]; };
  auto stage_sig = [&]() {
    _Pragma("unroll 8") for (int i = tid; i < L * W; i += kT) sig_sh[i] = __ldg(sig + i);
    sig = sig_sh;
  };
  if (!kLong) {
    stage_sig();
    unsigned long long* ks = reinterpret_cast<unsigned long long*>(arena);        // dead once the important set is marked
    if (a.keys) {
      _Pragma("unroll 8") for (int i = tid; i < L; i += kT) ks[i] = keys[i];
    } else {
      const double* imp = a.imp + (size_t)layer * s.T + t0;
      _Pragma("unroll 8") for (int i = tid; i < L; i += kT) ks[i] = importance_key(__ldg(imp + i), i, L, a.keep_initial, a.keep_recent);
    }
    keys = ks;
  }
  const int n_words = (L + 31) >> 5;
  int r_lo, r_hi;                            // contiguous token range of this warp
  sel::warp_range<kT>(L, warp, r_lo, r_hi);

  for (int i = tid; i < n_words; i += kT) { imp_mask[i] = 0; rep_mask[i] = 0; }
  __syncthreads();

  // ---- 1. important tokens: the b_imp largest keys, ties to the lower index --------------------
  if (b_imp > 0) sel::mark_top_keys<kT>(keys, L, b_imp, imp_mask, sc, kLong ? sig_sh : nullptr);

  // ---- 2-4. representatives of the other tokens ------------------------------------------------
  if (b_rep > 0) {
    const int N = L - b_imp;
    if (kLong && sig_sh) { stage_sig(); __syncthreads(); }
    // anchor
    if (a.anchor_mode == KVCRUSH_ANCHOR_MEAN) {
      for (int i = tid; i < 128; i += kT) bit_cnt[i] = 0;
      __syncthreads();
      int acc[4] = {0, 0, 0, 0};
      for (int base = r_lo; base < r_hi; base += 32) {
        const int i = base + lane;
        const bool cand = i < r_hi && !((imp_mask[base >> 5] >> lane) & 1u);
        _Pragma("unroll") for (int w = 0; w < W; ++w) {
          const uint32_t word = cand ? sig[(size_t)i * W + w] : 0u;
          const int nb = min(32, s.Hq - 32 * w);
          for (int b = 0; b < nb; ++b) {
            const unsigned m = __ballot_sync(kFull, (word >> b) & 1u);
            if (lane == b) acc[w] += __popc(m);
          }
        }
      }
      _Pragma("unroll") for (int w = 0; w < W; ++w)
        if (32 * w + lane < s.Hq && acc[w]) atomicAdd(&bit_cnt[32 * w + lane], acc[w]);
      __syncthreads();
      if (warp < W) {
        const int h = 32 * warp + lane;
        const unsigned word = __ballot_sync(kFull, h < s.Hq && 2LL * bit_cnt[h] >= N);
        if (lane == 0) anchor_sh[warp] = word;
      }
    } else if (tid < W) {
      uint32_t word;
      if (a.anchor_mode == KVCRUSH_ANCHOR_EXPLICIT)
        word = __ldg(a.anchor_bits + (a.anchor_per_segment ? (size_t)seg * W : 0) + tid);
      else
        word = 0xAAAAAAAAu;
      anchor_sh[tid] = word & head_mask(s.Hq, tid);
    }
    for (int i = tid; i < kWarps * kMaxBins; i += kT) (&warp_hist[0][0])[i] = 0;
    __syncthreads();
    uint32_t anc[4], hm[4];
    _Pragma("unroll") for (int w = 0; w < 4; ++w) { anc[w] = w < W ? anchor_sh[w] : 0u; hm[w] = w < W ? head_mask(s.Hq, w) : 0u; }
    const int n_bins = s.Hq + 1;

    // counting sort by (d, t): per-warp histograms over contiguous token ranges.  When there is room, the first
    // sweep also notes every token's distance and its position among the warp's tokens of that distance, so that
    // the second sweep is a plain scatter; otherwise the first sweep only counts.
    for (int base = r_lo; base < r_hi; base += 32) {
      const int i = base + lane;
      const bool cand = i < r_hi && !((imp_mask[base >> 5] >> lane) & 1u);
      int d = 0;
      if (cand)
        _Pragma("unroll") for (int w = 0; w < W; ++w) d += __popc((sig[(size_t)i * W + w] ^ anc[w]) & hm[w]);
      if (kLong) {
        if (cand) atomicAdd(&warp_hist[warp][d], 1);
        continue;
      }
      const unsigned voters = __ballot_sync(kFull, cand);
      unsigned peers = 0;
      if (cand) {
        peers = __match_any_sync(voters, d);
        sort_code[i] = (uint32_t)d | ((uint32_t)(warp_hist[warp][d] + __popc(peers & lt_mask)) << 8);
      } else if (i < r_hi) {
        sort_code[i] = 0xFFFFFFFFu;
      }
      __syncwarp();
      if (cand && (peers & lt_mask) == 0) warp_hist[warp][d] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    if (tid < n_bins) {                     // per bin: exclusive prefix over warps (token order)
      int run = 0;
      for (int w = 0; w < kWarps; ++w) { const int c = warp_hist[w][tid]; warp_hist[w][tid] = run; run += c; }
      bin_base[tid + 1] = run;
    }
    __syncthreads();
    if (tid == 0) {
      bin_base[0] = 0;
      for (int b = 1; b <= n_bins; ++b) bin_base[b] += bin_base[b - 1];
    }
    __syncthreads();
    if (!kLong) {
      for (int i = r_lo + lane; i < r_hi; i += 32) {
        const uint32_t c = sort_code[i];
        if (c != 0xFFFFFFFFu) {
          const int d = (int)(c & 0xFFu);
          sorted[bin_base[d] + warp_hist[warp][d] + (int)(c >> 8)] = i;
        }
      }
    } else {
      for (int base = r_lo; base < r_hi; base += 32) {
        const int i = base + lane;
        const bool cand = i < r_hi && !((imp_mask[base >> 5] >> lane) & 1u);
        int d = 0;
        if (cand)
          _Pragma("unroll") for (int w = 0; w < W; ++w) d += __popc((sig[(size_t)i * W + w] ^ anc[w]) & hm[w]);
        const unsigned voters = __ballot_sync(kFull, cand);
        unsigned peers = 0;
        if (cand) {
          peers = __match_any_sync(voters, d);
          const int pos = bin_base[d] + warp_hist[warp][d] + __popc(peers & lt_mask);
          if (sorted16) sorted16[pos] = (uint16_t)i; else sorted[pos] = i;
        }
        __syncwarp();
        if (cand && (peers & lt_mask) == 0) warp_hist[warp][d] += __popc(peers);
        __syncwarp();
      }
    }
    __syncthreads();

    // one representative per equal-frequency bucket
    // bucket i covers sorted positions [floor(i*N/R), floor((i+1)*N/R)); N = q_nr*R + r_nr
    const int q_nr = N / b_rep, r_nr = N - q_nr * b_rep;
    const int m_max = q_nr + (r_nr > 0 ? 1 : 0);                               // largest bucket
    if (m_max <= 16) {
      // Small buckets (the usual case: N/R is the compression ratio): 32 / gw buckets share a warp, one lane per member.
      // sum_{h set in t} n_h = sum over members u of popc(sig_t & sig_u), so
      // cost(t) = m * popc(sig_t) - 2 * sum_u popc(sig_t & sig_u): gw shuffles inside the lane group.
      // |cost| <= 16 * 128 and t < 2^18, so (cost, t) packs into 31 bits and one warp-level minimum per lane group
      // picks the representative, ties to the lower token.  The step is bound by its shuffles and bit counts, so the group
      // width follows the bucket closer than the next power of two in long segments (32768 tokens, 3277 buckets of 9: 74
      // thousand cycles with 16 lanes, 57 with 10; in short ones the wider choice of code costs more than it gives).
      const int gw = m_max <= 2 ? 2 : m_max <= 4 ? 4 : kLong && m_max <= 6 ? 6 : m_max <= 8 ? 8 : kLong && m_max <= 10 ? 10 : 16;
      const int per_warp = 32 / gw, sub = lane / gw, j = lane - sub * gw, g0 = sub * gw;   // sub == per_warp: lanes left over
      const unsigned gmask = sub < per_warp ? (0xFFFFFFFFu >> (32 - gw)) << g0 : 0xFFFFFFFFu << g0;
      // bucket b starts at b*q_nr + frac with b*r_nr = frac*R + rem.  Divisions are slow, so each lane divides once
      // for its first bucket and then steps exactly by the warp's stride of kWarps*per_warp buckets.
      const int first_bkt = warp * per_warp + sub, stride_b = kWarps * per_warp;
      const unsigned long long p0 = (unsigned long long)(unsigned)first_bkt * (unsigned)r_nr;
      const unsigned long long ps = (unsigned long long)(unsigned)stride_b * (unsigned)r_nr;
      int frac = (int)(p0 / (unsigned)b_rep), rem = (int)(p0 - (unsigned long long)frac * (unsigned)b_rep);
      const int step_q = (int)(ps / (unsigned)b_rep), step_r = (int)(ps - (unsigned long long)step_q * (unsigned)b_rep);
      for (int bkt = first_bkt; bkt - sub < b_rep; bkt += stride_b) {
        const bool live = sub < per_warp && bkt < b_rep;
        const int lo = live ? bkt * q_nr + frac : 0;
        const int m = live ? q_nr + (rem + r_nr >= b_rep ? 1 : 0) : 0;       // the next bucket's frac is one larger
        frac += step_q;
        rem += step_r;
        if (rem >= b_rep) { rem -= b_rep; ++frac; }
        const bool member = j < m;
        const int t = member ? sorted_at(lo + j) : 0;
        uint32_t mine[4] = {0u, 0u, 0u, 0u};
        _Pragma("unroll") for (int w = 0; w < W; ++w) mine[w] = member ? sig[(size_t)t * W + w] & head_mask(s.Hq, w) : 0u;
        int ones = 0;
        _Pragma("unroll") for (int w = 0; w < W; ++w) ones += __popc(mine[w]);
        // lanes past a bucket's last member hold zeros and add nothing
        int common;
        if (gw == 8) common = group_and_popc<W, 8>(mine, g0);
        else if (gw == 4) common = group_and_popc<W, 4>(mine, g0);
        else if (gw == 2) common = group_and_popc<W, 2>(mine, g0);
        else if (kLong && gw == 6) common = group_and_popc<W, 6>(mine, g0);
        else if (kLong && gw == 10) common = group_and_popc<W, 10>(mine, g0);
        else common = group_and_popc<W, 16>(mine, g0);
        const int cost = m * ones - 2 * common;
        const uint32_t key = member ? ((uint32_t)(cost + 4096) << 18) | (uint32_t)t : 0xFFFFFFFFu;
        const uint32_t best = __reduce_min_sync(gmask, key);
        if (j == 0 && live) {
          const uint32_t bt = best & 0x3FFFFu;
          atomicOr(&rep_mask[bt >> 5], 1u << (bt & 31));
        }
      }
    } else {
    // Larger buckets: one warp per bucket.  64-bit divisions are slow, so each
    // warp divides once and then steps exactly: i*N = pos*R + rem, and the stride kWarps*N = step_q*R + step_r.
    const long long stride = (long long)kWarps * N;
    const int step_q = (int)(stride / b_rep), step_r = (int)(stride - (long long)step_q * b_rep);
    int pos = (int)(((long long)warp * N) / b_rep);
    int rem = (int)((long long)warp * N - (long long)pos * b_rep);
    for (int bkt = warp; bkt < b_rep; bkt += kWarps) {
      const int lo = pos;
      const int hi = pos + q_nr + (rem + r_nr >= b_rep ? 1 : 0);
      const int m = hi - lo;
      pos += step_q;
      rem += step_r;
      if (rem >= b_rep) { rem -= b_rep; ++pos; }
      unsigned long long best = ~0ull;
      if (m <= 32) {
        // one lane per member.  sum_{h set in t} n_h = sum over members u of popc(sig_t & sig_u), so
        // cost(t) = m * popc(sig_t) - 2 * sum_u popc(sig_t & sig_u): m shuffles instead of one ballot per head
        const bool member = lane < m;
        const int t = member ? sorted_at(lo + lane) : 0;
        uint32_t mine[4] = {0u, 0u, 0u, 0u};
        _Pragma("unroll") for (int w = 0; w < W; ++w) mine[w] = member ? sig[(size_t)t * W + w] & head_mask(s.Hq, w) : 0u;
        int ones = 0, shared = 0;
        _Pragma("unroll") for (int w = 0; w < W; ++w) ones += __popc(mine[w]);
        for (int u0 = 0; u0 < m; u0 += 4) {        // lanes >= m hold zeros, so reading past m adds nothing
          _Pragma("unroll") for (int du = 0; du < 4; ++du)
            _Pragma("unroll") for (int w = 0; w < W; ++w) shared += __popc(mine[w] & __shfl_sync(kFull, mine[w], (u0 + du) & 31));
        }
        const int cost = m * ones - 2 * shared;
        if (member) best = ((unsigned long long)((uint32_t)cost + 0x80000000u) << 32) | (uint32_t)t;
      } else {
        int n_ones[4] = {0, 0, 0, 0};        // lane b of word w holds n_h for head 32w+b
        for (int c0 = lo; c0 < hi; c0 += 32) {
          const bool member = c0 + lane < hi;
          const int t = member ? sorted_at(c0 + lane) : 0;
          _Pragma("unroll") for (int w = 0; w < W; ++w) {
            const uint32_t word = member ? sig[(size_t)t * W + w] : 0u;
            const int nb = min(32, s.Hq - 32 * w);
            for (int b = 0; b < nb; ++b) {
              const unsigned ones = __ballot_sync(kFull, (word >> b) & 1u);
              if (lane == b) n_ones[w] += __popc(ones);
            }
          }
        }
        for (int c0 = lo; c0 < hi; c0 += 32) {
          const bool member = c0 + lane < hi;
          const int t = member ? sorted_at(c0 + lane) : 0;
          int cost = 0;
          _Pragma("unroll") for (int w = 0; w < W; ++w) {
            const uint32_t word = member ? sig[(size_t)t * W + w] : 0u;
            const int nb = min(32, s.Hq - 32 * w);
            for (int b = 0; b < nb; ++b) {
              const int n_h = __shfl_sync(kFull, n_ones[w], b);
              if ((word >> b) & 1u) cost += m - 2 * n_h;
            }
          }
          if (member) {
            const unsigned long long key = ((unsigned long long)((uint32_t)cost + 0x80000000u) << 32) | (uint32_t)t;
            best = key < best ? key : best;
          }
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(kFull, best, d);
        best = o < best ? o : best;
      }
      if (lane == 0) {
        const uint32_t t = (uint32_t)best;
        atomicOr(&rep_mask[t >> 5], 1u << (t & 31));
      }
    }
    }
    __syncthreads();
  }

  // ---- 5. kept = important U representatives, ascending ------------------------------------------
  sel::emit_kept<kT>(imp_mask, rep_mask, n_words, out_idx, out_kind, sc);
}

// ---- the same selection by a cluster of C blocks, for few long segments ------------------------------------------
// One block takes a long segment's chain of steps alone while most of the chip idles.  Here every block owns a contiguous
// range of the tokens (keys, signatures, masks) and a range of the buckets; what they exchange goes through distributed
// shared memory: extremes and histogram of the keys, the few candidates at the k-th largest, counts of the distances, the
// tokens and signatures in (d, t) order - each sent straight to the block that owns its bucket, so that the bucket step
// reads its signatures in order - and the representatives' bits.  Eight cluster barriers as a rule (start, key range, histogram,
// candidates, distances, order, representatives, counts), one more each for a mean anchor and for a tie that is cut, two more
// for every further radix round (more than 256 candidates).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() { cluster_arrive(); cluster_wait(); }
// the same shared variable in block `rank` of the cluster
template <class T>
__device__ __forceinline__ T* peer_of(T* p, int rank) {
  T* d;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(d) : "l"(p), "r"(rank));
  return d;
}

template <int W, int C, int kT>
__global__ void __launch_bounds__(kT, 1)
select_cluster_kernel(Shape s, SelectArgs a) {
  constexpr int kWarps = kT / 32;
  extern __shared__ __align__(16) uint32_t dyn_smem[];
  __shared__ sel::Scratch sc;                        // own histogram and candidates, read by the peers
  __shared__ alignas(16) uint32_t hist[sel::kBins];  // of the whole segment
  __shared__ unsigned long long list[sel::kRankList];
  __shared__ int warp_hist[kWarps][kMaxBins];
  __shared__ int bin_base[kMaxBins];
  __shared__ int bit_cnt[128];
  __shared__ uint32_t anchor_sh[4];
  // one entry of every block
  __shared__ uint32_t all_range[C][2];
  __shared__ int all_bins[C][kMaxBins];
  __shared__ int all_bits[C][128];
  __shared__ int all_equal[C], all_kept[C];
  cluster_arrive();                                  // (waited for below: all blocks have started)
  chain_wait();                                      // (chain_trigger: at the end)

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int rank = blockIdx.x % C, seg = blockIdx.x / C;
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  const int t0 = __ldg(s.cu_seqlens + seq);
  const int L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int b_imp = max(0, __ldg(a.budget_imp + seg));
  const int b_rep = max(0, __ldg(a.budget_rep + seg));
  int32_t* out_idx = a.idx + __ldg(a.cu_kept + seg);
  uint8_t* out_kind = a.kind ? a.kind + __ldg(a.cu_kept + seg) : nullptr;

  if (a.n_kept && tid == 0 && rank == 0) a.n_kept[seg] = (int)min((long long)b_imp + b_rep, (long long)L);
  if ((long long)b_imp + b_rep >= L) {               // budget covers the sequence: keep everything
    for (int i = rank * kT + tid; i < L; i += C * kT) {
      out_idx[i] = i;
      if (out_kind) out_kind[i] = 0;
    }
    cluster_wait();
    return;
  }

  // tokens [c_lo, c_lo + n) of the segment are this block's; `per` is a multiple of 32
  const int per = ((L + C - 1) / C + 31) & ~31;
  const int c_lo = min(L, rank * per), n = min(L, c_lo + per) - c_lo;
  const int cap = a.stage_words;                     // tokens of a block of the longest segment, rounded up to 32
  uint32_t* imp_mask = dyn_smem;
  uint32_t* rep_mask = imp_mask + cap / 32;
  uint32_t* sig_sh = rep_mask + cap / 32;            // [cap][W]
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(sig_sh + cap * W);      // [cap], dead once the important set is marked
  uint32_t* sort_code = reinterpret_cast<uint32_t*>(keys);                                 // [cap]
  int32_t* sorted = reinterpret_cast<int32_t*>(sort_code + cap);                           // [cap]: this block's part of the (d, t) order ..
  uint32_t* sorted_sig = reinterpret_cast<uint32_t*>(sorted + cap);                        // [cap][W]: .. and the signatures

  const uint32_t* sig = a.sigs + ((size_t)layer * s.T + t0 + c_lo) * W;
  uint32_t lo32 = 0xFFFFFFFFu, hi32 = 0u;
  auto stage = [&](auto&& load) {
    for (int i0 = tid; i0 < n; i0 += 4 * kT) {
      unsigned long long v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = load(min(i0 + j * kT, n - 1));
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j * kT < n) {
          keys[i0 + j * kT] = v[j];
          lo32 = min(lo32, (uint32_t)(v[j] >> 32));
          hi32 = max(hi32, (uint32_t)(v[j] >> 32));
        }
    }
  };
  _Pragma("unroll 4") for (int i = tid; i < n * W; i += kT) sig_sh[i] = __ldg(sig + i);
  if (a.keys) {
    const unsigned long long* src = a.keys + (size_t)layer * s.T + t0 + c_lo;
    stage([&](int i) { return src[i]; });
  } else {
    const double* src = a.imp + (size_t)layer * s.T + t0 + c_lo;
    stage([&](int i) { return importance_key(__ldg(src + i), c_lo + i, L, a.keep_initial, a.keep_recent); });
  }
  const int n_words = (n + 31) >> 5;
  for (int i = tid; i < n_words; i += kT) { imp_mask[i] = 0; rep_mask[i] = 0; }
  for (int i = tid; i < sel::kBins; i += kT) sc.hist[i] = 0;
  if (tid == 0) sc.small_n = 0;
  lo32 = __reduce_min_sync(kFull, lo32);
  hi32 = __reduce_max_sync(kFull, hi32);
  if (lane == 0) sc.red[warp] = (unsigned long long)hi32 << 32 | lo32;
  __syncthreads();
  int r_lo, r_hi;                                    // contiguous token range of this warp
  sel::warp_range<kT>(n, warp, r_lo, r_hi);
  cluster_wait();

  // ---- 1. important tokens: the b_imp largest keys, ties to the lower index --------------------
  if (b_imp > 0) {
    if (warp == 0) {
      const unsigned long long v = sc.red[lane < kWarps ? lane : 0];
      lo32 = __reduce_min_sync(kFull, (uint32_t)v);
      hi32 = __reduce_max_sync(kFull, (uint32_t)(v >> 32));
      if (lane < C) {
        uint32_t* out = peer_of(&all_range[rank][0], lane);
        out[0] = lo32;
        out[1] = hi32;
      }
    }
    cluster_barrier();
    lo32 = 0xFFFFFFFFu; hi32 = 0u;
#pragma unroll
    for (int c = 0; c < C; ++c) { lo32 = min(lo32, all_range[c][0]); hi32 = max(hi32, all_range[c][1]); }
    // radix rounds over x = key - base, base = the smallest upper half with zeros below: x has `rem` significant bits; `top`
    // is the value of the bits of x above them chosen so far
    const unsigned long long base = (unsigned long long)lo32 << 32;
    int rem = 32 + (hi32 > lo32 ? 32 - __clz(hi32 - lo32) : 0);
    unsigned long long top = 0;
    uint32_t k_rem = (uint32_t)b_imp, n_equal = 0;
    for (bool first = true; rem > 0; first = false) {
      const int w = min(rem, sel::kDigitBits), shift = rem - w, n_bins = 1 << w;
      for (int i = tid; i < n; i += kT) {
        const unsigned long long x = keys[i] - base;
        if (first || (x >> rem) == top) atomicAdd(&sc.hist[(uint32_t)(x >> shift) & (uint32_t)(n_bins - 1)], 1u);
      }
      cluster_barrier();
      for (int i = tid; i < n_bins; i += kT) {
        uint32_t sum = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) sum += peer_of(sc.hist, c)[i];
        hist[i] = sum;
      }
      __syncthreads();
      sel::find_digit_desc<kT>(hist, n_bins, k_rem, sc.warp_tot, sc.sel);
      top = (top << w) | sc.sel[0];
      k_rem = sc.sel[1];
      n_equal = sc.sel[2];
      rem = shift;
      if (rem == 0) break;
      if (n_equal <= (uint32_t)sel::kRankList) {     // few candidates: every block ranks all of them
        for (int i = tid; i < n; i += kT) {
          const unsigned long long x = keys[i] - base;
          if ((x >> rem) == top) sc.small[atomicAdd(&sc.small_n, 1u)] = x;
        }
        cluster_barrier();
        int at = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const int m = (int)*peer_of(&sc.small_n, c);
          const unsigned long long* from = peer_of(sc.small, c);
          for (int i = tid; i < m; i += kT) list[at + i] = from[i];
          at += m;
        }
        __syncthreads();
        if (tid < at) {
          const unsigned long long v = list[tid];
          uint32_t gt = 0, ge = 0;
#pragma unroll 4
          for (int j = 0; j < at; ++j) {
            const unsigned long long o = list[j];
            gt += o > v;
            ge += o >= v;
          }
          if (gt < k_rem && k_rem <= ge) { sc.sel_x = v; sc.sel[1] = k_rem - gt; sc.sel[2] = ge - gt; }   // equal candidates agree
        }
        __syncthreads();
        top = sc.sel_x;
        k_rem = sc.sel[1];
        n_equal = sc.sel[2];
        break;
      }
      cluster_barrier();                             // the peers have read this histogram
      for (int i = tid; i < sel::kBins; i += kT) sc.hist[i] = 0;
      __syncthreads();
    }
    const unsigned long long kth = base + top;
    int eq_before = 0;
    const bool cut = k_rem != n_equal;               // a tie is cut: tokens equal to the k-th largest are admitted in order
    if (cut) {
      int n_eq = 0;
      for (int i = r_lo + lane; i < r_hi; i += 32) n_eq += keys[i] == kth;
      n_eq = __reduce_add_sync(kFull, n_eq);
      __syncthreads();                               // warp_tot may still be read by the digit search
      if (lane == 0) sc.warp_tot[warp] = n_eq;
      __syncthreads();
      if (warp == 0) {
        const int total = __reduce_add_sync(kFull, lane < kWarps ? sc.warp_tot[lane] : 0);
        if (lane < C) *peer_of(&all_equal[rank], lane) = total;
      }
      eq_before = sel::warps_before(sc.warp_tot, warp, lane);
      cluster_barrier();
      for (int c = 0; c < rank; ++c) eq_before += all_equal[c];
    }
    for (int base_i = r_lo; base_i < r_hi; base_i += 32) {
      const int i = base_i + lane;
      const unsigned long long key = i < r_hi ? keys[i] : 0ull;
      bool imp = i < r_hi && key >= kth;
      if (cut) {
        const bool eq = imp && key == kth;
        const unsigned eq_b = __ballot_sync(kFull, eq);
        imp = imp && (!eq || (uint32_t)(eq_before + __popc(eq_b & lt_mask)) < k_rem);
        eq_before += __popc(eq_b);
      }
      const unsigned imp_b = __ballot_sync(kFull, imp);
      if (lane == 0) imp_mask[base_i >> 5] = imp_b;
    }
    __syncthreads();
  }

  // ---- 2-4. representatives of the other tokens ------------------------------------------------
  if (b_rep > 0) {
    const int N = L - b_imp;
    if (a.anchor_mode == KVCRUSH_ANCHOR_MEAN) {
      for (int i = tid; i < 128; i += kT) bit_cnt[i] = 0;
      __syncthreads();
      int acc[4] = {0, 0, 0, 0};
      for (int base = r_lo; base < r_hi; base += 32) {
        const int i = base + lane;
        const bool cand = i < r_hi && !((imp_mask[base >> 5] >> lane) & 1u);
        _Pragma("unroll") for (int w = 0; w < W; ++w) {
          const uint32_t word = cand ? sig_sh[(size_t)i * W + w] : 0u;
          const int nb = min(32, s.Hq - 32 * w);
          for (int b = 0; b < nb; ++b) {
            const unsigned m = __ballot_sync(kFull, (word >> b) & 1u);
            if (lane == b) acc[w] += __popc(m);
          }
        }
      }
      _Pragma("unroll") for (int w = 0; w < W; ++w)
        if (32 * w + lane < s.Hq && acc[w]) atomicAdd(&bit_cnt[32 * w + lane], acc[w]);
      __syncthreads();
      for (int i = tid; i < 128 * C; i += kT) *peer_of(&all_bits[rank][i & 127], i >> 7) = bit_cnt[i & 127];
      cluster_barrier();
      if (warp < W) {
        const int h = 32 * warp + lane;
        long long cnt = 0;
        _Pragma("unroll") for (int c = 0; c < C; ++c) cnt += all_bits[c][h];
        const unsigned word = __ballot_sync(kFull, h < s.Hq && 2 * cnt >= N);
        if (lane == 0) anchor_sh[warp] = word;
      }
    } else if (tid < W) {
      uint32_t word;
      if (a.anchor_mode == KVCRUSH_ANCHOR_EXPLICIT)
        word = __ldg(a.anchor_bits + (a.anchor_per_segment ? (size_t)seg * W : 0) + tid);
      else
        word = 0xAAAAAAAAu;
      anchor_sh[tid] = word & head_mask(s.Hq, tid);
    }
    for (int i = tid; i < kWarps * kMaxBins; i += kT) (&warp_hist[0][0])[i] = 0;
    __syncthreads();
    uint32_t anc[4], hm[4];
    _Pragma("unroll") for (int w = 0; w < 4; ++w) { anc[w] = w < W ? anchor_sh[w] : 0u; hm[w] = w < W ? head_mask(s.Hq, w) : 0u; }
    const int n_bins = s.Hq + 1;

    // counting sort by (d, t): every token's distance and its position among the warp's tokens of that distance
    for (int base = r_lo; base < r_hi; base += 32) {
      const int i = base + lane;
      const bool cand = i < r_hi && !((imp_mask[base >> 5] >> lane) & 1u);
      int d = 0;
      if (cand)
        _Pragma("unroll") for (int w = 0; w < W; ++w) d += __popc((sig_sh[(size_t)i * W + w] ^ anc[w]) & hm[w]);
      const unsigned voters = __ballot_sync(kFull, cand);
      unsigned peers = 0;
      if (cand) {
        peers = __match_any_sync(voters, d);
        sort_code[i] = (uint32_t)d | ((uint32_t)(warp_hist[warp][d] + __popc(peers & lt_mask)) << 8);
      } else if (i < r_hi) {
        sort_code[i] = 0xFFFFFFFFu;
      }
      __syncwarp();
      if (cand && (peers & lt_mask) == 0) warp_hist[warp][d] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // per bin: exclusive prefix over the warps (token order); the block's totals go to everybody
    for (int b = warp; b < n_bins; b += kWarps) {
      const int c = lane < kWarps ? warp_hist[lane][b] : 0;
      int incl = c;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += v;
      }
      if (lane < kWarps) warp_hist[lane][b] = incl - c;
      const int total = __shfl_sync(kFull, incl, 31);
      if (lane < C) *peer_of(&all_bins[rank][b], lane) = total;
    }
    cluster_barrier();
    if (warp == 0) {                                 // start of every bin: lower bins of all blocks, this bin of lower blocks
      int run = 0;
      for (int b0 = 0; b0 < n_bins; b0 += 32) {
        const int b = b0 + lane;
        int before = 0, total = 0;
        if (b < n_bins)
          _Pragma("unroll") for (int c = 0; c < C; ++c) { const int v = all_bins[c][b]; total += v; before += c < rank ? v : 0; }
        int incl = total;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int v = __shfl_up_sync(kFull, incl, d);
          if (lane >= d) incl += v;
        }
        if (b < n_bins) bin_base[b] = run + incl - total + before;
        run += __shfl_sync(kFull, incl, 31);
      }
    }
    __syncthreads();

    // Block c owns the buckets [b_rep * c / C, b_rep * (c + 1) / C) and with them the sorted positions from start[c].  Where
    // fewer buckets than blocks make one part longer than `cap`, the order goes through global memory instead.
    auto bucket_of = [&](int c) { return (int)((long long)b_rep * c / C); };
    int start[C + 1], longest = 0;
#pragma unroll
    for (int c = 0; c <= C; ++c) {
      start[c] = (int)((long long)bucket_of(c) * N / b_rep);
      if (c > 0) longest = max(longest, start[c] - start[c - 1]);
    }
    const bool local = longest <= cap;
    int32_t* sorted_g = a.sorted + (size_t)layer * s.T + t0;
    for (int i = r_lo + lane; i < r_hi; i += 32) {
      const uint32_t code = sort_code[i];
      if (code == 0xFFFFFFFFu) continue;
      const int d = (int)(code & 0xFFu), pos = bin_base[d] + warp_hist[warp][d] + (int)(code >> 8);
      if (!local) { sorted_g[pos] = c_lo + i; continue; }
      int o = 0, first = 0;
#pragma unroll
      for (int c = 1; c < C; ++c)
        if (pos >= start[c]) { o = c; first = start[c]; }
      *peer_of(sorted + (pos - first), o) = c_lo + i;
      _Pragma("unroll") for (int w = 0; w < W; ++w)
        *peer_of(sorted_sig + (size_t)(pos - first) * W + w, o) = sig_sh[(size_t)i * W + w] & hm[w];
    }
    cluster_barrier();
    const uint32_t* sig_g = a.sigs + ((size_t)layer * s.T + t0) * W;
    int own_start = 0;
#pragma unroll
    for (int c = 1; c < C; ++c)
      if (rank == c) own_start = start[c];
    const int b_lo = bucket_of(rank), b_hi = bucket_of(rank + 1);
    auto token_at = [&](int p) { return local ? sorted[p - own_start] : __ldcg(sorted_g + p); };
    auto sig_at = [&](int p, int t, int w) { return local ? sorted_sig[(size_t)(p - own_start) * W + w] : __ldg(sig_g + (size_t)t * W + w) & hm[w]; };
    auto mark = [&](uint32_t t) {
      const uint32_t o = t / (uint32_t)per, i = t - o * per;
      atomicOr(peer_of(rep_mask, (int)o) + (i >> 5), 1u << (i & 31));
    };

    // one representative per equal-frequency bucket: bucket b covers the positions [floor(b N / R), floor((b + 1) N / R))
    const int q_nr = N / b_rep, r_nr = N - q_nr * b_rep;
    const int m_max = q_nr + (r_nr > 0 ? 1 : 0);                                // largest bucket
    if (m_max <= 16) {
      // 32 / gw buckets share a warp, one lane per member: see select_segment_kernel
      const int gw = m_max <= 2 ? 2 : m_max <= 4 ? 4 : m_max <= 6 ? 6 : m_max <= 8 ? 8 : m_max <= 10 ? 10 : 16;
      const int per_warp = 32 / gw, sub = lane / gw, j = lane - sub * gw, g0 = sub * gw;   // sub == per_warp: lanes left over
      const unsigned gmask = sub < per_warp ? (0xFFFFFFFFu >> (32 - gw)) << g0 : 0xFFFFFFFFu << g0;
      const int first_bkt = b_lo + warp * per_warp + sub, stride_b = kWarps * per_warp;
      const unsigned long long p0 = (unsigned long long)(unsigned)first_bkt * (unsigned)r_nr;
      const unsigned long long ps = (unsigned long long)(unsigned)stride_b * (unsigned)r_nr;
      int frac = (int)(p0 / (unsigned)b_rep), rem = (int)(p0 - (unsigned long long)frac * (unsigned)b_rep);
      const int step_q = (int)(ps / (unsigned)b_rep), step_r = (int)(ps - (unsigned long long)step_q * (unsigned)b_rep);
      for (int bkt = first_bkt; bkt - sub < b_hi; bkt += stride_b) {
        const bool live = sub < per_warp && bkt < b_hi;
        const int lo = live ? bkt * q_nr + frac : 0;
        const int m = live ? q_nr + (rem + r_nr >= b_rep ? 1 : 0) : 0;
        frac += step_q;
        rem += step_r;
        if (rem >= b_rep) { rem -= b_rep; ++frac; }
        const bool member = j < m;
        const int t = member ? token_at(lo + j) : 0;
        uint32_t mine[4] = {0u, 0u, 0u, 0u};
        int ones = 0;
        _Pragma("unroll") for (int w = 0; w < W; ++w) { mine[w] = member ? sig_at(lo + j, t, w) : 0u; ones += __popc(mine[w]); }
        int common;
        if (gw == 8) common = group_and_popc<W, 8>(mine, g0);
        else if (gw == 4) common = group_and_popc<W, 4>(mine, g0);
        else if (gw == 2) common = group_and_popc<W, 2>(mine, g0);
        else if (gw == 6) common = group_and_popc<W, 6>(mine, g0);
        else if (gw == 10) common = group_and_popc<W, 10>(mine, g0);
        else common = group_and_popc<W, 16>(mine, g0);
        // |cost| <= 16 * 128 and t < 2^18: (cost, t) packs into 31 bits
        const uint32_t key = member ? ((uint32_t)(m * ones - 2 * common + 4096) << 18) | (uint32_t)t : 0xFFFFFFFFu;
        const uint32_t best = __reduce_min_sync(gmask, key);
        if (j == 0 && live) mark(best & 0x3FFFFu);
      }
    } else {
      // larger buckets: a warp per bucket; lane b of word w counts the members with bit 32 w + b set
      for (int b = b_lo + warp; b < b_hi; b += kWarps) {
        const long long x = (long long)b * r_nr;
        const int frac = (int)(x / b_rep), rem = (int)(x - (long long)frac * b_rep);
        const int lo = b * q_nr + frac, m = q_nr + (rem + r_nr >= b_rep ? 1 : 0);
        int n_ones[4] = {0, 0, 0, 0};
        for (int u = 0; u < m; u += 32) {
          const bool member = u + lane < m;
          const int t = member && !local ? token_at(lo + u + lane) : 0;
          _Pragma("unroll") for (int w = 0; w < W; ++w) {
            const uint32_t word = member ? sig_at(lo + u + lane, t, w) : 0u;
            const int nb = min(32, s.Hq - 32 * w);
            for (int i = 0; i < nb; ++i) {
              const unsigned ones = __ballot_sync(kFull, (word >> i) & 1u);
              if (lane == i) n_ones[w] += __popc(ones);
            }
          }
        }
        unsigned long long best = ~0ull;
        for (int u = 0; u < m; u += 32) {
          const bool member = u + lane < m;
          const int t = member ? token_at(lo + u + lane) : 0;
          int cost = 0;
          _Pragma("unroll") for (int w = 0; w < W; ++w) {
            const uint32_t word = member ? sig_at(lo + u + lane, t, w) : 0u;
            const int nb = min(32, s.Hq - 32 * w);
            for (int i = 0; i < nb; ++i) {
              const int n_h = __shfl_sync(kFull, n_ones[w], i);
              if ((word >> i) & 1u) cost += m - 2 * n_h;
            }
          }
          if (member) {
            const unsigned long long key = ((unsigned long long)((uint32_t)cost + 0x80000000u) << 32) | (uint32_t)t;
            best = key < best ? key : best;
          }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
          const unsigned long long o = __shfl_xor_sync(kFull, best, d);
          best = o < best ? o : best;
        }
        if (lane == 0) mark((uint32_t)best);
      }
    }
    cluster_barrier();
  }

  // ---- 5. kept = important U representatives, ascending ------------------------------------------
  int cnt = 0;
  for (int i = tid; i < n_words; i += kT) cnt += __popc(imp_mask[i] | rep_mask[i]);
  cnt = __reduce_add_sync(kFull, cnt);
  __syncthreads();
  if (lane == 0) sc.warp_tot[warp] = cnt;
  __syncthreads();
  if (warp == 0) {
    const int total = __reduce_add_sync(kFull, lane < kWarps ? sc.warp_tot[lane] : 0);
    if (lane < C) *peer_of(&all_kept[rank], lane) = total;
  }
  chain_trigger();                                   // blocks of the next kernel, set up earlier, would crowd on the SMs without a cluster
  cluster_barrier();                                 // from here on nobody touches a peer's memory
  int before = 0;
  for (int c = 0; c < rank; ++c) before += all_kept[c];
  sel::emit_kept<kT>(imp_mask, rep_mask, n_words, out_idx + before, out_kind ? out_kind + before : nullptr, sc, c_lo);
}

}  // namespace

int launch_importance(const Shape& s, const float* scores, int keep_initial, int keep_recent,
                      unsigned long long* keys, cudaStream_t stream) {
  const size_t n = (size_t)s.n_layers * s.T;
  return launch_chained(importance_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, stream, 1, s, scores, keep_initial,
                        keep_recent, keys);
}

int launch_importance_keys(const Shape& s, const double* importance, int keep_initial, int keep_recent,
                           unsigned long long* keys, cudaStream_t stream) {
  const size_t n = (size_t)s.n_layers * s.T;
  return launch_chained(importance_keys_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, stream, 1, s, importance,
                        keep_initial, keep_recent, keys);
}

namespace {

constexpr int kClusterSmem = 180 * 1024;           // dynamic shared memory select_cluster_kernel may take (static part: ~46 KB)
int cluster_tokens(const Shape& s, int cluster) { return ((s.max_seqlen + cluster - 1) / cluster + 31) & ~31; }
size_t cluster_bytes(const Shape& s, int cap) { return (size_t)cap / 4 + (size_t)cap * (8 + 8 * s.W); }

// Blocks of a segment's cluster, 0: one block by itself.  A cluster pays from about 8192 tokens on, where the step is more
// work than barriers, and while its blocks find SMs (about 33 clusters of four, 15 of eight).  One block / cluster of 4 / of 8:
// 1 segment of 4096 tokens 13.6 / 15.0 / 15.3 us, of 8192 19.2 / 17.9 / 17.9, of 16384 36.4 / 22.6 / 22.5, of 32768 65.8 / 32.0 /
// 26.7; 8 of 20000 51.1 / 29.3 / 26.7; 32 of 4096 14.1 / 16.4 / 46, of 8192 19.5 / 19.2 / 53, of 16384 38.6 / 24.0 / 68, of 32768
// 70.7 / 34.1 / 81.  Twice as many take two rounds of half the time: 36 of 8192 19.6 / 35.7, but 64 of 32768 74.8 / 67.1, of 25000
// 60.9 / 56.2.  The longest segment decides in ragged batches as well: one of 30000 and 60 of 1000 62.4 / 30.3, 64 between 1000 and
// 32768 70.6 / 60.7, 64 between 8000 and 25000 57.0 / 52.6, one of 12300 and 15 of 500 33.1 / 20.4 (whole selection, 8 heads).
// held(c): the device runs clusters of c such blocks at all.
template <class Held>
int select_cluster_size(const Shape& s, long long n_seg, int n_sms, Held&& held) {
  auto fits = [&](int c) { return cluster_bytes(s, cluster_tokens(s, c)) <= (size_t)kClusterSmem; };
  const bool few = n_seg * 8 <= n_sms * 4 / 5;
  if (s.max_seqlen < (few ? 8192 : 12288)) return 0;
  if (s.max_seqlen > 16384 && few && fits(8) && held(8)) return 8;
  if (n_seg * 4 <= n_sms * (s.max_seqlen > 24576 ? 7 / 4.0 : 7 / 8.0) && fits(4) && held(4)) return 4;
  return 0;
}

template <int W, int C>
constexpr auto cluster_kernel = select_cluster_kernel<W, C, 1024>;

// Whether this device runs a cluster of C blocks with all the shared memory they may take (write-once cache per device: the
// answer depends on nothing else).
template <int W, int C>
bool holds_cluster() {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> known[kMaxDevices];                  // 1: yes, 2: no
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return false; }
  if (const int k = known[dev].load(std::memory_order_relaxed)) return k == 1;
  if (allow_dynamic_smem(cluster_kernel<W, C>, kClusterSmem) != KVCRUSH_OK) return false;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = kClusterSmem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, cluster_kernel<W, C>, &cfg) != cudaSuccess) { cudaGetLastError(); return false; }
  known[dev].store(n > 0 ? 1 : 2, std::memory_order_relaxed);
  return n > 0;
}
bool holds_cluster(int words, int cluster) {
  switch (words) {
    case 1: return cluster == 4 ? holds_cluster<1, 4>() : holds_cluster<1, 8>();
    case 2: return cluster == 4 ? holds_cluster<2, 4>() : holds_cluster<2, 8>();
    case 3: return cluster == 4 ? holds_cluster<3, 4>() : holds_cluster<3, 8>();
    default: return cluster == 4 ? holds_cluster<4, 4>() : holds_cluster<4, 8>();
  }
}

}  // namespace

int select_blocks_of_a_segment(const Shape& s, int n_sms, int largest_cluster) {
  const int n = select_cluster_size(s, (long long)s.n_layers * s.n_seqs, n_sms, [&](int c) { return c <= largest_cluster; });
  return n > 0 ? n : 1;
}

size_t select_workspace_bytes(const Shape& s) {
  const size_t n = (size_t)s.n_layers * s.T;
  return ((n * 8 + 255) / 256) * 256 + ((n * 4 + 255) / 256) * 256;
}

int launch_select(const Shape& s, const float* scores, const double* importance, const uint32_t* sigs,
                  const int32_t* budget_imp,
                  const int32_t* budget_rep, int anchor_mode, const uint32_t* anchor_bits, int anchor_per_segment,
                  int keep_initial, int keep_recent, const int32_t* cu_kept, int32_t* idx, uint8_t* kind,
                  int32_t* n_kept, void* ws, cudaStream_t stream) {
  if (s.T == 0) {                                   // nothing but empty sequences: every segment keeps nothing
    if (n_kept && cudaMemsetAsync(n_kept, 0, (size_t)s.n_layers * s.n_seqs * sizeof(int32_t), stream) != cudaSuccess)
      return KVCRUSH_ERR_CUDA;
    return KVCRUSH_OK;
  }
  const size_t n = (size_t)s.n_layers * s.T;
  unsigned long long* keys = static_cast<unsigned long long*>(ws);
  int32_t* sorted = reinterpret_cast<int32_t*>(static_cast<unsigned char*>(ws) + ((n * 8 + 255) / 256) * 256);

  SelectArgs a{};
  a.sigs = sigs; a.budget_imp = budget_imp; a.budget_rep = budget_rep;
  a.anchor_mode = anchor_mode; a.anchor_bits = anchor_bits; a.anchor_per_segment = anchor_per_segment;
  a.cu_kept = cu_kept; a.idx = idx; a.kind = kind; a.n_kept = n_kept; a.sorted = sorted;
  a.mask_words = ((s.max_seqlen + 31) / 32 + 3) & ~3;
  a.stage_words = (s.max_seqlen + 3) & ~3;
  size_t dyn = (size_t)a.mask_words * 2 * sizeof(uint32_t);
  const size_t budget = 208 * 1024;     // dynamic shared memory this kernel may take (static part: ~18 KB)
  const size_t per_tok = (size_t)a.stage_words * sizeof(uint32_t);
  const bool long_seg = dyn + per_tok * (s.W + 3) > budget;
  if (!long_seg) {
    dyn += per_tok * (s.W + 3);
  } else {
    if (dyn + per_tok * s.W <= budget) { a.stage_sig = 1; dyn += per_tok * s.W; }
    if (s.max_seqlen <= 65536 && dyn + per_tok / 2 <= budget) { a.stage_sorted = 1; dyn += per_tok / 2; }
  }
  const long long n_seg = (long long)s.n_layers * s.n_seqs;
  const int n_sms = sm_count();
  const int cluster = select_cluster_size(s, n_seg, n_sms, [&](int c) { return holds_cluster(s.W, c); });
  // importance keys: computed here from the scores, or taken from the caller's I(t) - converted while the segment
  // kernel stages them, or by a small kernel when the segments are too long to be staged
  if (!importance) {
    if (launch_importance(s, scores, keep_initial, keep_recent, keys, stream) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
    a.keys = keys;
  }
  if (importance) {
    if (!long_seg || cluster > 0) {
      a.imp = importance; a.keep_initial = keep_initial; a.keep_recent = keep_recent;
    } else {
      if (launch_importance_keys(s, importance, keep_initial, keep_recent, keys, stream) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
      a.keys = keys;
    }
  }
  if (cluster > 0) {
    const int cap = cluster_tokens(s, cluster);
    const size_t cluster_dyn = cluster_bytes(s, cap);
    a.stage_words = cap;
    auto launch = [&](auto kern) {
      if (allow_dynamic_smem(kern, kClusterSmem) != KVCRUSH_OK) return (int)KVCRUSH_ERR_CUDA;
      return launch_chained(kern, dim3((unsigned)(n_seg * cluster)), dim3(1024), cluster_dyn, stream, cluster, s, a);
    };
    auto by_words = [&](auto w) {
      constexpr int W = decltype(w)::value;
      return cluster == 4 ? launch(cluster_kernel<W, 4>) : launch(cluster_kernel<W, 8>);
    };
    return s.W == 1 ? by_words(std::integral_constant<int, 1>{}) : s.W == 2 ? by_words(std::integral_constant<int, 2>{})
         : s.W == 3 ? by_words(std::integral_constant<int, 3>{}) : by_words(std::integral_constant<int, 4>{});
  }
  auto launch = [&](auto kern, int threads) {
    // static + dynamic shared memory above the 48 KB default needs the opt-in
    if (dyn > 28 * 1024 && allow_dynamic_smem(kern, (int)budget) != KVCRUSH_OK) return (int)KVCRUSH_ERR_CUDA;
    return launch_chained(kern, dim3((unsigned)(s.n_layers * s.n_seqs)), dim3(threads), dyn, stream, 1, s, a);
  };
  // Threads of a segment: 1024 while every segment has an SM to itself (32 x 8192 tokens 22 us, with 512 threads 27), half as
  // many up to 1024 tokens, where barriers are most of the work (one segment of 512 tokens 7.7 -> 6.7 us, with 256 threads
  // 7.5).  Registers let an SM hold 1024 threads, so more segments than SMs take smaller blocks as far as shared memory
  // holds them: 256 segments of 700 tokens 17.2 -> 10.6 us, 224 of 1900 21.6 -> 15.4, 512 of 4000 62.7 -> 48.1 (with 256
  // threads 60.7); 512 of 700 tokens 31.9 -> 13.0 (18.9), 512 of 1900 42.0 -> 23.7 (28.6).
  auto resident = [&](int n) { return n * (dyn + 19 * 1024) <= 227 * 1024; };
  auto by_words = [&](auto w) {
    constexpr int W = decltype(w)::value;
    if (long_seg) return launch(select_segment_kernel<W, true, 1024>, 1024);
    if (n_seg > 2 * n_sms && s.max_seqlen <= 2048 && resident(4)) return launch(select_segment_kernel<W, false, 256>, 256);
    if ((s.max_seqlen <= 1024 || n_seg > n_sms) && resident(2)) return launch(select_segment_kernel<W, false, 512>, 512);
    return launch(select_segment_kernel<W, false, 1024>, 1024);
  };
  return s.W == 1 ? by_words(std::integral_constant<int, 1>{}) : s.W == 2 ? by_words(std::integral_constant<int, 2>{})
       : s.W == 3 ? by_words(std::integral_constant<int, 3>{}) : by_words(std::integral_constant<int, 4>{});
}

}  // namespace kvc

// Stage 1 on CUDA cores (fp32 arithmetic): attention column sums (Algorithm 1 of the paper,
// "attention weights" and "normalized attention score" steps).  Serves fp32 inputs and shapes the
// tensor-core kernels do not cover (bf16 and fp16 inputs are widened on load); the S x S matrix is never stored.
//
// Two sweeps of one tiled kernel: row log-sum-exps, then column sums.  64 x 64 logit tiles from fp32 copies of both
// operands in shared memory, 4 x 4 logits a thread, so that a 16-byte shared-memory read feeds eight FMAs (one warp
// per row and one dot product per lane spent 170 us on 8 heads x 512 tokens of 64 channels, all of it waiting for loads,
// and 2174 us on 4 layers of 1024 tokens; the two sweeps now take 26 and 190 us).  Of a call of few blocks the column sweep
// stages its tiles and forms its first logits while the row sweep ends: whole pass of 8 heads x 512 tokens 45.2 -> 40.0 us, with
// operands that no cache holds 47.7 -> 41.3.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace kvc {

namespace {

namespace cg = cooperative_groups;

constexpr int kRows = 64;                    // rows of both operands' tiles
constexpr int kThreads = 256;
constexpr int kMaxD = 256;

// kPastL1: a kernel that may read the operands before it waits for the one in front (see common.cuh).
template <bool kPastL1, class V>
__device__ __forceinline__ V load(const V* p) { if constexpr (kPastL1) return __ldcg(p); else return __ldg(p); }

template <bool kPastL1>
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = load<kPastL1>(reinterpret_cast<const float4*>(p));
  const float4 b = load<kPastL1>(reinterpret_cast<const float4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

template <bool kPastL1>
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 r = load<kPastL1>(reinterpret_cast<const uint4*>(p));
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

template <bool kPastL1>
__device__ __forceinline__ void load8(const __half* p, float (&v)[8]) {
  const uint4 r = load<kPastL1>(reinterpret_cast<const uint4*>(p));
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
    v[2 * i] = f.x;
    v[2 * i + 1] = f.y;
  }
}

// Rows of a [kRows][D] tile start kPad floats apart from a multiple of 32 banks, so that the 16-byte reads of 16
// consecutive rows do not meet in a bank.
constexpr int kPad = 4;

// Stages rows row0 .. row0+kStaged-1 of a sequence of L tokens (zeros past its end) as fp32.
template <typename T, int kStaged, bool kPastL1>
__device__ __forceinline__ void stage_tile(float* sh, const T* base, long long stride, int row0, int L, int D) {
  const int vec = D / 8;                                    // 8 channels at a time
  for (int e = threadIdx.x; e < kStaged * vec; e += kThreads) {
    const int r = e / vec, d = (e - r * vec) * 8;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (row0 + r < L) load8<kPastL1>(base + (long long)(row0 + r) * stride + d, v);
    float4* out = reinterpret_cast<float4*>(sh + r * (D + kPad) + d);
    out[0] = make_float4(v[0], v[1], v[2], v[3]);
    out[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// One sweep over the logits.  A cluster owns kRows rows of the stationary operand of one (layer, head, sequence); its
// blocks take the streamed operand's tiles in turn, and block 0 adds up what they found (through distributed shared
// memory, in the order of the blocks).
//   kColsum = false   stationary queries, streamed keys: (max, sum of 2^(x - max)) of every query row
//   kColsum = true    stationary keys, streamed queries: sum of 2^(x - lse2(query)) of every key
// 256 threads as 16 x 16; a thread holds N x N logits of a tile: 4 x 4, or 1 x 1 or 2 x 2 where no sequence is longer than
// 16 or 32 tokens and the rest of the 64 x 64 would be zeros (300 sequences of 5 tokens, 2 layers x 8 heads: 237 -> 70 us).
// kLate: the column sweep takes the row log-sum-exp behind a tile's products instead of beside its loads, so that it can start
// while the row sweep ends (`early`).  Tiles of 64 x 64 do so in any case, which costs nothing there (100 sequences of 300 tokens
// 1062 -> 1048 us, 8 heads x 8192 tokens 2394 -> 2382, 32 heads x 1024 of 128 channels 343.6 -> 347.4); smaller ones, a product
// of a few steps between two barriers, only where they start early (300 sequences of 5 tokens 66.2 -> 64.2 us without).
// Grid: (slot, layer, head) x the cluster's blocks.  In a batch of sequences of similar length slots are (tile, sequence)
// pairs, the heaviest tiles of all sequences first (4 layers x 8 heads x 6 sequences of 600 tokens: 424 us, sequence by sequence
// 453).  Otherwise (by_seq) sequence i owns the slots cu[i] / kRows + i up to the next one's first: at least as many as it has
// tiles, and in all only T / kRows + n_seqs of them, found without a table.
template <typename T, bool kColsum, int N, bool kLate>
__global__ void __launch_bounds__(kThreads)
simt_sweep_kernel(Shape s, TensorView Q, TensorView K, float scale_log2, const float* __restrict__ lse, float lse_mul,
                  float* __restrict__ lse2_out, float* __restrict__ lse_nat_out, float* __restrict__ scores, int normalize,
                  int layer0, int n_layers, int by_seq, int early) {
  extern __shared__ float4 dyn4[];
  float* fix_sh = reinterpret_cast<float*>(dyn4);
  float* str_sh = fix_sh + 16 * N * (s.D + kPad);
  __shared__ float part[2][kRows];                          // this block's maximum (sweep 1) and sum of every row
  __shared__ float nlse_sh[kRows];                          // sweep 2: minus lse2 of the streamed queries that vote
  if (!kLate || !early) {                                   // early: sweep 1 of the same call is the launch before
    chain_wait();
    chain_trigger();
  }
  cg::cluster_group cluster = cg::this_cluster();
  const int n_blk = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  int unit = blockIdx.x / n_blk;
  const int h = unit % s.Hq; unit /= s.Hq;
  const int layer = layer0 + unit % n_layers; unit /= n_layers;
  int seq = 0;                                              // unit is the slot
  if (!by_seq) {
    seq = unit % s.n_seqs;
  } else {
    for (int end = s.n_seqs; end - seq > 1;) {              // the last sequence whose first slot is not above it
      const int mid = (seq + end) >> 1;
      if (__ldg(s.cu_seqlens + mid) / kRows + mid <= unit) seq = mid; else end = mid;
    }
  }
  const int t0 = __ldg(s.cu_seqlens + seq), L = __ldg(s.cu_seqlens + seq + 1) - t0;
  const int rank_tile = by_seq ? unit - (t0 / kRows + seq) : unit / s.n_seqs;
  const int n_tiles = (L + kRows - 1) / kRows;
  if (rank_tile >= n_tiles) return;                         // uniform over the cluster, like every exit below
  // heaviest tiles first: the last query rows, the first keys
  const int tile = kColsum ? rank_tile : n_tiles - 1 - rank_tile;
  const int row0 = tile * kRows;
  const int ws = (s.window > 0 && L > s.window) ? L - s.window : 0;       // first voting query
  if (!kColsum && row0 + kRows <= ws) return;               // no query of this tile votes
  const int first = kColsum ? max(s.causal ? tile : 0, ws / kRows) : 0;
  const int last = kColsum ? n_tiles : (s.causal ? tile + 1 : n_tiles);   // streamed tiles [first, last)
  const T* qbase = static_cast<const T*>(Q.ptr) + layer * Q.sl + (long long)t0 * Q.st + h * Q.sh;
  const T* kbase = static_cast<const T*>(K.ptr) + layer * K.sl + (long long)t0 * K.st + (h / s.G) * K.sh;
  const size_t vec0 = ((size_t)layer * s.Hq + h) * s.T + t0;
  const float ninf = -INFINITY;

  stage_tile<T, 16 * N, kLate || N == 4>(fix_sh, kColsum ? kbase : qbase, kColsum ? K.st : Q.st, row0, L, s.D);
  float m[N], sum[N];
#pragma unroll
  for (int i = 0; i < N; ++i) { m[i] = ninf; sum[i] = 0.f; }
  for (int u = first + rank; u < last; u += n_blk) {
    __syncthreads();                                        // the previous tile is done with
    stage_tile<T, 16 * N, kLate || N == 4>(str_sh, kColsum ? qbase : kbase, kColsum ? Q.st : K.st, u * kRows, L, s.D);
    if (kColsum && !kLate && tid < kRows) {
      const int j = u * kRows + tid;
      nlse_sh[tid] = j < L && j >= ws ? -(__ldcg(lse + vec0 + j) * lse_mul) : ninf;
    }
    __syncthreads();
    float acc[N][N];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) acc[i][j] = 0.f;
    const float* fa = fix_sh + ty * (s.D + kPad);           // stationary rows ty + 16 i, streamed rows tx + 16 j
    const float* fb = str_sh + tx * (s.D + kPad);
#pragma unroll 2
    for (int d = 0; d < s.D; d += 4) {
      float4 a[N], b[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        a[i] = *reinterpret_cast<const float4*>(fa + i * 16 * (s.D + kPad) + d);
        b[i] = *reinterpret_cast<const float4*>(fb + i * 16 * (s.D + kPad) + d);
      }
#pragma unroll
      for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j)
          acc[i][j] = fmaf(a[i].w, b[j].w, fmaf(a[i].z, b[j].z, fmaf(a[i].y, b[j].y, fmaf(a[i].x, b[j].x, acc[i][j]))));
    }
    if constexpr (kLate) {                                  // the row log-sum-exp is needed only now
      if (early && u == first + rank) {
        chain_wait();
        chain_trigger();
      }
      if (tid < kRows) {
        const int j = u * kRows + tid;
        nlse_sh[tid] = j < L && j >= ws ? -(__ldcg(lse + vec0 + j) * lse_mul) : ninf;
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int r = row0 + ty + 16 * i;
      float x[4] = {ninf, ninf, ninf, ninf};
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int c = u * kRows + tx + 16 * j;
        // a query before the window may share the tile: its logits are left out whatever they are (inf and NaN included)
        const bool in = c < L && (!kColsum || c >= ws) && (!s.causal || (kColsum ? c >= r : c <= r));
        x[j] = in ? (kColsum ? fmaf(acc[i][j], scale_log2, nlse_sh[tx + 16 * j]) : acc[i][j] * scale_log2) : ninf;
      }
      if constexpr (kColsum) {
        sum[i] += (exp2f(x[0]) + exp2f(x[1])) + (exp2f(x[2]) + exp2f(x[3]));
      } else {
        const float big = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        if (big > m[i]) { sum[i] *= exp2f(m[i] - big); m[i] = big; }     // first tile: 0 * 2^-inf
        const float ref = m[i] == ninf ? 0.f : m[i];                     // no maximum yet: -inf adds 0, NaN makes the sum NaN
        sum[i] += (exp2f(x[0] - ref) + exp2f(x[1] - ref)) + (exp2f(x[2] - ref) + exp2f(x[3] - ref));
      }
    }
  }
  // the 16 threads of a row, then the blocks of the cluster
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float big = m[i];
    if constexpr (!kColsum) {
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) big = fmaxf(big, __shfl_xor_sync(0xFFFFFFFFu, big, d));
      sum[i] = sum[i] == 0.f ? 0.f : sum[i] * exp2f(m[i] - big);           // 0: nothing seen
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) sum[i] += __shfl_xor_sync(0xFFFFFFFFu, sum[i], d);
    if (tx == 0) { part[0][ty + 16 * i] = big; part[1][ty + 16 * i] = sum[i]; }
  }
  if (n_blk > 1) cluster.sync(); else __syncthreads();
  if (rank == 0 && tid < 16 * N && row0 + tid < L) {
    const size_t out = vec0 + row0 + tid;
    float big = ninf, total = 0.f;
    if constexpr (!kColsum)
      for (int b = 0; b < n_blk; ++b) big = fmaxf(big, *cluster.map_shared_rank(&part[0][tid], b));
    for (int b = 0; b < n_blk; ++b) {
      const float p = *cluster.map_shared_rank(&part[1][tid], b);
      total += kColsum ? p : p == 0.f ? 0.f : p * exp2f(*cluster.map_shared_rank(&part[0][tid], b) - big);
    }
    if constexpr (kColsum) {
      scores[out] = normalize ? total / (float)(L - ws) : total;
    } else if (row0 + tid >= ws) {
      const float v = big + log2f(total);
      lse2_out[out] = v;
      if (lse_nat_out) lse_nat_out[out] = v * 0.69314718055994530942f;
    }
  }
  if (n_blk > 1) cluster.sync();                            // block 0 has read the others' parts
}

template <typename T, bool kColsum, int N>
int launch_sweep(const Shape& s, const int32_t* cu_host, const TensorView& Q, const TensorView& K, float scale_log2, const float* lse, float lse_mul,
                 float* lse2_out, float* lse_nat_out, float* scores, int normalize, bool early, cudaStream_t stream) {
  const int max_tiles = (s.max_seqlen + kRows - 1) / kRows;
  long long tiles = 0;
  for (int i = 0; i < s.n_seqs; ++i) tiles += (cu_host[i + 1] - cu_host[i] + kRows - 1) / kRows;
  const long long units = tiles * s.n_layers * s.Hq;
  // A small problem does not fill the chip with one block per tile of rows: its streamed tiles are shared by up to 8
  // blocks then (8 heads x 512 tokens: 64 tiles of rows, 4 blocks each; with 8 the second wave starts, 26 -> 37 us).
  const int n_sms = sm_count();
  int n_blk = 1;
  while (n_blk < 8 && 2 * n_blk <= max_tiles && units * n_blk < n_sms) n_blk *= 2;
  const long long pairs = (long long)max_tiles * s.n_seqs;
  const int by_seq = 8 * pairs > 9 * tiles;
  const long long slots = by_seq ? (long long)s.T / kRows + s.n_seqs : pairs, per_layer = slots * s.Hq * n_blk;
  if (per_layer > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  const size_t dyn = (size_t)2 * 16 * N * (s.D + kPad) * sizeof(float);
  // Blocks that are set up while the predecessor still runs are placed where there is room first, not evenly.  A grid of more
  // than a block an SM pays for that unless its blocks are short: 2 layers x 8 heads, 500 + 300 + 700 tokens, both sweeps 146
  // against 109 us; 8 heads x 512 tokens, two tiles a block, whole pass 46 against 47 us.
  const int streamed = s.window > 0 && s.window / kRows + 2 < max_tiles ? s.window / kRows + 2 : max_tiles;
  const bool overlap = per_layer * s.n_layers <= n_sms || (per_layer * s.n_layers <= 2 * n_sms && streamed <= 2 * n_blk);
  early = early && overlap;                                 // (one launch then)
  auto kern = kColsum && (N == 4 || early) ? simt_sweep_kernel<T, kColsum, N, kColsum> : simt_sweep_kernel<T, kColsum, N, kColsum && N == 4>;
  if (dyn > 40 * 1024 && allow_dynamic_smem(kern, 2 * 16 * N * (kMaxD + kPad) * (int)sizeof(float)) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
  const int layers = (int)(0x7FFFFFFFLL / per_layer < s.n_layers ? 0x7FFFFFFFLL / per_layer : s.n_layers);    // of one launch
  for (int layer0 = 0; layer0 < s.n_layers; layer0 += layers) {
    const int n = s.n_layers - layer0 < layers ? s.n_layers - layer0 : layers;
    const int rc = launch_kernel(overlap, kern, dim3((unsigned)(per_layer * n)), dim3(kThreads), dyn, stream, n_blk, s, Q, K, scale_log2,
                                  lse, lse_mul, lse2_out, lse_nat_out, scores, normalize, layer0, n, by_seq, early);
    if (rc != KVCRUSH_OK) return rc;
  }
  return KVCRUSH_OK;
}

template <typename T, int N>
int run_tiles(const Shape& s, const int32_t* cu_host, const TensorView& Q, const TensorView& K, float scale_log2, const float* lse_in,
              float lse_in_mul, float* lse2_ws, float* scores, float* lse_out, int normalize, cudaStream_t stream) {
  if (!lse_in) {
    const int rc = launch_sweep<T, false, N>(s, cu_host, Q, K, scale_log2, nullptr, 1.f, lse2_ws, lse_out, nullptr, 0, false, stream);
    if (rc != KVCRUSH_OK) return rc;
    return launch_sweep<T, true, N>(s, cu_host, Q, K, scale_log2, lse2_ws, 1.f, nullptr, nullptr, scores, normalize, true, stream);
  }
  return launch_sweep<T, true, N>(s, cu_host, Q, K, scale_log2, lse_in, lse_in_mul, nullptr, nullptr, scores, normalize, false, stream);
}

template <typename T>
int run(const Shape& s, const int32_t* cu_host, const TensorView& Q, const TensorView& K, float scale_log2, const float* lse_in,
        float lse_in_mul, float* lse2_ws, float* scores, float* lse_out, int normalize, cudaStream_t stream) {
  if (s.T == 0) return KVCRUSH_OK;
  auto kern = s.max_seqlen <= 16 ? run_tiles<T, 1> : s.max_seqlen <= 32 ? run_tiles<T, 2> : run_tiles<T, 4>;
  return kern(s, cu_host, Q, K, scale_log2, lse_in, lse_in_mul, lse2_ws, scores, lse_out, normalize, stream);
}

}  // namespace

int launch_score_simt(const Shape& s, const int32_t* cu_host, const TensorView& Q, const TensorView& K, float scale_log2,
                      const float* lse_in, float lse_in_mul, float* lse2_ws, float* scores, float* lse_out,
                      int normalize, int32_t* /*status*/, cudaStream_t stream) {
  if (s.D > kMaxD || s.D % 8 != 0) return KVCRUSH_ERR_UNSUPPORTED;
  if (Q.dtype == KVCRUSH_FP32)
    return run<float>(s, cu_host, Q, K, scale_log2, lse_in, lse_in_mul, lse2_ws, scores, lse_out, normalize, stream);
  if (Q.dtype == KVCRUSH_BF16)
    return run<__nv_bfloat16>(s, cu_host, Q, K, scale_log2, lse_in, lse_in_mul, lse2_ws, scores, lse_out, normalize, stream);
  if (Q.dtype == KVCRUSH_FP16)
    return run<__half>(s, cu_host, Q, K, scale_log2, lse_in, lse_in_mul, lse2_ws, scores, lse_out, normalize, stream);
  return KVCRUSH_ERR_UNSUPPORTED;
}

}  // namespace kvc

// Max pooling of the per-head scores along the token axis (SnapKV's way of keeping the neighbours of a
// high-scoring token, named in Sec. 2.3 / 4.1.1 of the paper): out[l][h][t] = max over the centred window of
// odd width `kernel`, clipped to t's own sequence.
//
// Bound by latency and by the two passes over the scores.  A block takes a chunk of 1024 tokens (256 when that
// would leave SMs idle: one layer of 700 + 300 tokens 2.6 -> 2.1 us; 1024 rows of 2000 tokens 11.5 against 6.5 us) of one
// (layer, head) row: it stages them and the window's overhang in shared memory, all loads in flight together, 16 bytes wide
// where the rows allow it.  Where then the chunk lies in one sequence, places outside the sequence hold NaN, which fmaxf passes over, and a thread takes four
// neighbouring outputs from 16-byte reads.  32 x 32 rows of 8192 tokens, width 7: 20 us against 42 us with one output a
// thread, whose window came from L1 behind a 64-bit division.
#include "common.cuh"

namespace kvc {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxChunk = 1024;

// kStaged: the chunk and its overhang (rounded up to whole quads) fit in shared memory.  quads: 16-byte accesses.
template <bool kStaged>
__global__ void __launch_bounds__(kThreads)
pool_scores_kernel(Shape s, const float* __restrict__ in, int radius, int chunk, int n_chunks, int quads, float* __restrict__ out) {
  extern __shared__ float4 stage4[];
  float* stage = reinterpret_cast<float*>(stage4);
  chain_wait();
  chain_trigger();
  const int row = blockIdx.x / n_chunks, t0 = (blockIdx.x - row * n_chunks) * chunk, tid = threadIdx.x;
  const int t_end = min(t0 + chunk, s.T);
  const float* src = in + (size_t)row * s.T;
  float* dst = out + (size_t)row * s.T;
  int first = max(t0 - radius, 0);                               // stage[0] is the row's element `first`
  bool staged = false;
  if constexpr (kStaged) {
    if (quads) {
      const int pad = (radius + 3) / 4, n_quads = chunk / 4 + 2 * pad, q0 = t0 / 4 - pad;    // stage4[0] is the row's quad q0
      float4 v[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int q = q0 + tid + j * kThreads;
        v[j] = tid + j * kThreads < n_quads && q >= 0 && 4 * q < s.T ? __ldg(reinterpret_cast<const float4*>(src) + q) : float4{};
      }
      const int seq = seq_of_token(s.cu_seqlens, s.n_seqs, t0);
      const int a = __ldg(s.cu_seqlens + seq), b = __ldg(s.cu_seqlens + seq + 1);
      auto stage_all = [&](auto&& put) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (tid + j * kThreads < n_quads) put(tid + j * kThreads, v[j]);
        for (int i = tid + 2 * kThreads; i < n_quads; i += kThreads) {
          const int q = q0 + i;
          put(i, q >= 0 && 4 * q < s.T ? __ldg(reinterpret_cast<const float4*>(src) + q) : float4{});
        }
        __syncthreads();
      };
      if (t_end <= b) {
        stage_all([&](int i, float4 x) {
          const int t = 4 * (q0 + i);
          const float none = __int_as_float(0x7FFFFFFF);
          if (t < a || t >= b) x.x = none;
          if (t + 1 < a || t + 1 >= b) x.y = none;
          if (t + 2 < a || t + 2 >= b) x.z = none;
          if (t + 3 < a || t + 3 >= b) x.w = none;
          stage4[i] = x;
        });
        if (t0 + 4 * tid >= t_end) return;
        float m[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) m[j] = __int_as_float(0x7FFFFFFF);
        for (int c = 0; c <= 2 * pad; ++c) {                      // quad c covers offsets e .. e + 3 from the first output
          const float4 x = stage4[tid + c];
          const int e = 4 * (c - pad);
          if (e >= 3 - radius && e + 3 <= radius) {               // in all four windows
            const float y = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
#pragma unroll
            for (int j = 0; j < 4; ++j) m[j] = fmaxf(m[j], y);
          } else {
            const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (abs(e + i - j) <= radius) m[j] = fmaxf(m[j], xs[i]);
          }
        }
        reinterpret_cast<float4*>(dst)[t0 / 4 + tid] = make_float4(m[0], m[1], m[2], m[3]);
        return;
      }
      stage_all([&](int i, float4 x) { stage4[i] = x; });
      first = 4 * q0;
      staged = true;
    }
  }
  int t = t0 + tid, seq = 0, seq_first = 0, seq_end = 0;
  if (t < t_end) {
    seq = seq_of_token(s.cu_seqlens, s.n_seqs, t);
    seq_first = __ldg(s.cu_seqlens + seq);
    seq_end = __ldg(s.cu_seqlens + seq + 1);
  }
  if constexpr (kStaged) {
    if (!staged) {
      const int last = min(t_end - 1 + radius, s.T - 1);
#pragma unroll 5
      for (int u = first + tid; u <= last; u += kThreads) stage[u - first] = __ldg(src + u);
      __syncthreads();
    }
  }
  auto at = [&](int u) { return kStaged ? stage[u - first] : __ldg(src + u); };
  for (; t < t_end; t += kThreads) {
    while (t >= seq_end) { seq_first = seq_end; seq_end = __ldg(s.cu_seqlens + ++seq + 1); }
    const int lo = max(seq_first, t - radius), hi = min(seq_end - 1, t + radius);
    float m = at(lo);
#pragma unroll 4
    for (int u = lo + 1; u <= hi; ++u) m = fmaxf(m, at(u));
    dst[t] = m;
  }
}

}  // namespace

int launch_pool_scores(const Shape& s, const float* scores_in, int kernel, float* scores_out, cudaStream_t stream) {
  const int radius = (kernel - 1) / 2;
  const long long rows = (long long)s.n_layers * s.Hq;
  const int chunk = rows * ((s.T + kMaxChunk - 1) / kMaxChunk) >= 8 * sm_count() ? kMaxChunk : kThreads;
  const int n_chunks = (s.T + chunk - 1) / chunk;
  const long long blocks = rows * n_chunks;
  if (blocks == 0) return KVCRUSH_OK;
  if (blocks > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  const long long staged = ((long long)chunk + 2LL * (radius / 4 + 1) * 4) * sizeof(float);
  const bool fits = staged <= 48 * 1024;
  const int quads = s.T % 4 == 0 && reinterpret_cast<uintptr_t>(scores_in) % 16 == 0 && reinterpret_cast<uintptr_t>(scores_out) % 16 == 0;
  return launch_chained(fits ? pool_scores_kernel<true> : pool_scores_kernel<false>, dim3((unsigned)blocks), dim3(kThreads),
                        fits ? (size_t)staged : 0, stream, 1, s, scores_in, radius, chunk, n_chunks, quads, scores_out);
}

}  // namespace kvc

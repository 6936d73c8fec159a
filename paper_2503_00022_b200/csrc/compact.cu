// Stage 4: gather of the kept K/V rows into the reduced cache (Sec. 3.2 of the paper: the
// representatives together with the important tokens form the final cache).
//
// Pure byte movement, bound by HBM bandwidth.  One warp owns one kept token of one layer and
// copies that token's rows of every KV head, for K and for V, as 16-byte vectors: the index
// arithmetic (segment search by the whole warp, source token) is paid once per token, and every lane
// keeps eight independent 16-byte loads of both tensors in flight before the first store.
// 512 segments x 21 pages of 32 tokens, 8 KV heads of 128: 411 us = 6.9 TB/s (495 us with a serial
// search, 64-bit divisions and one tensor after the other); one layer of 1024 tokens x 32 heads: 13.3 -> 7.5 us.
//
// Page-granular variant (Sec. 4.3.5: paged caches keep or drop whole pages): the kept list holds page numbers,
// a warp owns one token slot of one kept page, and the slots of a short last page are filled with zeros.
#include "common.cuh"

namespace kvc {

namespace {

constexpr int kWarpsPerBlock = 8;

struct CompactArgs {
  const unsigned char* src[2];
  unsigned char* dst[2];
  long long src_sl[2], src_st[2], src_sh[2];   // bytes
  long long dst_sl[2], dst_st[2], dst_sh[2];   // bytes
  int vec_per_row;                             // 16-byte vectors in one head row
  int n_vec;                                   // vectors per token = Hkv * vec_per_row
};

template <bool kPaged, int kTensors>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
compact_kernel(Shape s, CompactArgs a, const int32_t* __restrict__ cu_kept, const int32_t* __restrict__ idx,
               long long total_kept, int page_size) {
  chain_wait();
  chain_trigger();
  const int lane = threadIdx.x & 31;
  const long long out_row = (long long)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  // row = position in the kept list (a token, or a page of which this warp copies slot `slot`); 64-bit divisions are slow
  const long long row = !kPaged ? out_row : out_row <= 0x7FFFFFFF ? (long long)((unsigned)out_row / (unsigned)page_size) : out_row / page_size;
  const int slot = kPaged ? (int)(out_row - row * page_size) : 0;
  if (row >= total_kept) return;
  const int seg = warp_segment_of_row(cu_kept, s.n_layers * s.n_seqs, row, lane);
  const int layer = seg / s.n_seqs, seq = seg - layer * s.n_seqs;
  long long src_tok, dst_tok;
  bool present = true;
  if (kPaged) {
    const long long tok_in_seq = (long long)__ldg(idx + row) * page_size + slot;
    const int seq_begin = __ldg(s.cu_seqlens + seq);
    present = tok_in_seq < __ldg(s.cu_seqlens + seq + 1) - seq_begin;
    src_tok = seq_begin + tok_in_seq;
    dst_tok = (row - __ldg(cu_kept + layer * s.n_seqs)) * page_size + slot;
  } else {
    src_tok = (long long)__ldg(s.cu_seqlens + seq) + __ldg(idx + row);
    dst_tok = row - __ldg(cu_kept + layer * s.n_seqs);
  }

  // all loads of a step, of both tensors, are issued before the first store
  const unsigned char* sp[kTensors];
  unsigned char* dp[kTensors];
#pragma unroll
  for (int ten = 0; ten < kTensors; ++ten) {
    sp[ten] = a.src[ten] + layer * a.src_sl[ten] + src_tok * a.src_st[ten];
    dp[ten] = a.dst[ten] + layer * a.dst_sl[ten] + dst_tok * a.dst_st[ten];
  }
  for (int v0 = lane; v0 < a.n_vec; v0 += 4 * 32) {
    uint4 val[kTensors][4];
    int h[4], c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int v = v0 + u * 32;
      h[u] = v / a.vec_per_row;
      c[u] = v - h[u] * a.vec_per_row;
#pragma unroll
      for (int ten = 0; ten < kTensors; ++ten) {
        if (kPaged) val[ten][u] = make_uint4(0u, 0u, 0u, 0u);
        if (v < a.n_vec && (!kPaged || present))
          val[ten][u] = __ldcs(reinterpret_cast<const uint4*>(sp[ten] + h[u] * a.src_sh[ten]) + c[u]);
      }
    }
#pragma unroll
    for (int ten = 0; ten < kTensors; ++ten)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v0 + u * 32 < a.n_vec) __stcs(reinterpret_cast<uint4*>(dp[ten] + h[u] * a.dst_sh[ten]) + c[u], val[ten][u]);
  }
}

}  // namespace

namespace {

// Running scores follow the cache: out[l][h][dst] = in[l][h][src] for the kept tokens (or the slots of the kept
// pages; slots past the end of a sequence get 0).  One thread per (layer, kept row, group of 8 heads).
constexpr int kScoreHeads = 8;
__global__ void __launch_bounds__(256)
compact_scores_kernel(Shape s, const float* __restrict__ in, float* __restrict__ out, const int32_t* __restrict__ cu_kept,
                      const int32_t* __restrict__ idx, long long total_kept, int page_size, long long out_tokens) {
  chain_wait();
  chain_trigger();
  const long long out_row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const auto row_of = [&](long long r) {
    return r <= 0x7FFFFFFF ? (long long)((unsigned)r / (unsigned)page_size) : r / page_size;
  };
  const long long row = row_of(out_row), warp_row = row_of(out_row - lane);
  if (warp_row >= total_kept) return;                     // uniform over the warp
  const int n_seg = s.n_layers * s.n_seqs;
  int lo = warp_segment_of_row(cu_kept, n_seg, warp_row, lane);
  if (row >= total_kept) return;
  while (lo + 1 < n_seg && (long long)__ldg(cu_kept + lo + 1) <= row) ++lo;  // the warp's later rows may belong to a later segment
  const int slot = (int)(out_row - row * page_size);
  const int layer = lo / s.n_seqs, seq = lo - layer * s.n_seqs;
  const int seq_begin = __ldg(s.cu_seqlens + seq);
  const long long tok_in_seq = (long long)__ldg(idx + row) * page_size + slot;
  const bool present = tok_in_seq < __ldg(s.cu_seqlens + seq + 1) - seq_begin;
  const long long dst = (row - __ldg(cu_kept + layer * s.n_seqs)) * page_size + slot;
  // blockIdx.y takes every gridDim.y-th group of kScoreHeads heads: the loads of a group are in flight together
  const float* src = in + (long long)layer * s.Hq * s.T + seq_begin + tok_in_seq;
  float* dp = out + (long long)layer * s.Hq * out_tokens + dst;
  for (int h0 = blockIdx.y * kScoreHeads; h0 < s.Hq; h0 += gridDim.y * kScoreHeads) {
    float v[kScoreHeads];
#pragma unroll
    for (int j = 0; j < kScoreHeads; ++j)
      v[j] = present && h0 + j < s.Hq ? __ldg(src + (long long)(h0 + j) * s.T) : 0.f;
#pragma unroll
    for (int j = 0; j < kScoreHeads; ++j)
      if (h0 + j < s.Hq) dp[(long long)(h0 + j) * out_tokens] = v[j];
  }
}

int launch_gather(const Shape& s, const TensorView& K, const TensorView* V, int page_size, const int32_t* cu_kept,
                  const int32_t* idx, long long total_kept, const TensorView& K_out, const TensorView* V_out,
                  cudaStream_t stream) {
  if (total_kept == 0) return KVCRUSH_OK;
  const int eb = elt_bytes(K.dtype);
  CompactArgs a{};
  const int n_tensors = V ? 2 : 1;
  const TensorView* in[2] = {&K, V};
  const TensorView* out[2] = {&K_out, V_out};
  for (int i = 0; i < n_tensors; ++i) {
    a.src[i] = static_cast<const unsigned char*>(in[i]->ptr);
    a.dst[i] = static_cast<unsigned char*>(const_cast<void*>(out[i]->ptr));
    a.src_sl[i] = in[i]->sl * eb; a.src_st[i] = in[i]->st * eb; a.src_sh[i] = in[i]->sh * eb;
    a.dst_sl[i] = out[i]->sl * eb; a.dst_st[i] = out[i]->st * eb; a.dst_sh[i] = out[i]->sh * eb;
  }
  a.vec_per_row = s.D * eb / 16;
  a.n_vec = s.Hkv * a.vec_per_row;
  const long long rows = total_kept * (page_size > 0 ? page_size : 1);
  const long long blocks = (rows + kWarpsPerBlock - 1) / kWarpsPerBlock;
  if (blocks > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  auto kern = page_size > 0 ? (V ? compact_kernel<true, 2> : compact_kernel<true, 1>)
                            : (V ? compact_kernel<false, 2> : compact_kernel<false, 1>);
  return launch_chained(kern, dim3((unsigned)blocks), dim3(kWarpsPerBlock * 32), 0, stream, 1, s, a, cu_kept, idx, total_kept,
                        page_size > 0 ? page_size : 1);
}

}  // namespace

int launch_compact(const Shape& s, const TensorView& K, const TensorView* V, const int32_t* cu_kept,
                   const int32_t* idx, long long total_kept, const TensorView& K_out, const TensorView* V_out,
                   cudaStream_t stream) {
  return launch_gather(s, K, V, 0, cu_kept, idx, total_kept, K_out, V_out, stream);
}

int launch_compact_scores(const Shape& s, const float* scores_in, int page_size, const int32_t* cu_kept,
                          const int32_t* idx, long long total_kept, float* scores_out, long long out_tokens,
                          cudaStream_t stream) {
  if (total_kept == 0) return KVCRUSH_OK;
  const int ps = page_size > 0 ? page_size : 1;
  const long long rows = total_kept * ps;
  const long long blocks = (rows + 255) / 256;
  if (blocks > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  // In pages a thread takes more groups of heads where the rows alone fill the chip: consecutive rows are read together, and
  // finding a row costs as much as loading a group (16 x 736 tokens, 32 layers x 32 heads, pages of 32: 24.6 -> 19.9 us).  Single
  // tokens of a long cache are bound by their sectors and gain nothing (32768 tokens, a fifth kept: 26.0 -> 26.4).
  unsigned head_blocks = (unsigned)((s.Hq + kScoreHeads - 1) / kScoreHeads);
  while (ps > 1 && head_blocks > 1 && blocks * head_blocks > 16LL * sm_count()) head_blocks = (head_blocks + 1) / 2;
  const dim3 grid((unsigned)blocks, head_blocks);
  return launch_chained(compact_scores_kernel, grid, dim3(256), 0, stream, 1, s, scores_in, scores_out, cu_kept, idx, total_kept, ps,
                        out_tokens);
}

int launch_compact_pages(const Shape& s, const TensorView& K, const TensorView* V, int page_size,
                         const int32_t* cu_kept, const int32_t* page_idx, long long total_kept_pages,
                         const TensorView& K_out, const TensorView* V_out, cudaStream_t stream) {
  return launch_gather(s, K, V, page_size, cu_kept, page_idx, total_kept_pages, K_out, V_out, stream);
}

}  // namespace kvc

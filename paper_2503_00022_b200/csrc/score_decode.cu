// Decode step of stage 1 (Sec. 2.3 / 4.1.1 of the paper: H2O goes on summing attention weights while tokens are
// generated): every sequence has one new query, and its attention row over the sequence's cached keys is added to the
// running scores.
//
// Bound by reading K, which passes through the chip once: a cluster of 1 to 8 blocks shares one (layer, sequence, KV
// head), every block streams its part of the keys, keeps the logits of the group's query heads in shared memory, and
// the blocks exchange their (maximum, sum) pairs through distributed shared memory before each adds its part.
// Measured for 32 layers x 32 heads x 8192 keys: 345 us = 6.4 TB/s (1147 us when K was read twice by one thread per
// key); for 32 layers x 16 sequences of 680 keys, 8 KV heads of 4 query heads: 141 us = 5.7 TB/s (535 us).
//
// Tiles of 16 keys x 8 query heads go through mma.sync: the dot product may take the channels in any order, so a
// lane's 16-byte piece of a key row (8 channels) is used as the operand registers of two m16n8k16 steps as it arrives,
// with the query registers loaded in the same order - no staging, no shuffles, and a row's four lanes read 64
// consecutive bytes.  With one query head seven of the eight columns are idle, which costs nothing here: the tensor
// pipe is busy for a few per cent.  fp32 keys use the same tiles on the CUDA cores.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "common.cuh"

namespace kvc {

namespace {

namespace cg = cooperative_groups;

constexpr int kHeads = 8;                    // query heads of one pass over the keys
constexpr int kRows = 16;                    // keys of one tile
constexpr int kMaxCluster = 8;
constexpr int kMaxD = 256;
constexpr int kMaxStored = 200 * 1024;       // bytes of logits a block keeps in shared memory, at most
constexpr unsigned kAll = 0xFFFFFFFFu;

// One tile: keys t .. t+15 (rows beyond t_end read as zeros) against 8 heads.  Lane = 4 * g + c holds the pieces of keys g
// and g + 8 and gets their logits for heads 2c and 2c + 1: x[0], x[1] (key g), x[2], x[3] (key g + 8).
template <int DB>
struct Tile {
  uint4 a0[DB], a1[DB];
  template <typename T>
  __device__ __forceinline__ void load(const T* __restrict__ kbase, long long st, int t, int t_end, int D, int lane) {
    const int g = lane >> 2, c = lane & 3;
    const bool in0 = t + g < t_end, in1 = t + g + 8 < t_end;
    const T* r0 = kbase + (long long)(t + g) * st;
    const T* r1 = r0 + 8 * st;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < DB; ++i) {
      const int d = 32 * i + 8 * c;
      a0[i] = in0 && d < D ? __ldcs(reinterpret_cast<const uint4*>(r0 + d)) : zero;
      a1[i] = in1 && d < D ? __ldcs(reinterpret_cast<const uint4*>(r1 + d)) : zero;
    }
  }
  // qr: the lane's query registers, head g, channels 32 i + 8 c .. + 7
  template <typename T>
  __device__ __forceinline__ void logits(const uint4 (&qr)[DB], float (&x)[4]) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = 0.f;
#pragma unroll
    for (int i = 0; i < DB; ++i) {
#define KVC_MMA(TYPE, A0, A1, A2, A3, B0, B1)                                                                     \
  asm("mma.sync.aligned.m16n8k16.row.col.f32." TYPE "." TYPE ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};" \
      : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]) : "r"(A0), "r"(A1), "r"(A2), "r"(A3), "r"(B0), "r"(B1))
      if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        KVC_MMA("bf16", a0[i].x, a1[i].x, a0[i].y, a1[i].y, qr[i].x, qr[i].y);
        KVC_MMA("bf16", a0[i].z, a1[i].z, a0[i].w, a1[i].w, qr[i].z, qr[i].w);
      } else {
        KVC_MMA("f16", a0[i].x, a1[i].x, a0[i].y, a1[i].y, qr[i].x, qr[i].y);
        KVC_MMA("f16", a0[i].z, a1[i].z, a0[i].w, a1[i].w, qr[i].z, qr[i].w);
      }
#undef KVC_MMA
    }
  }
};

// The same tile of fp32 keys: a row's four lanes each take their channels for all 8 heads and add up by two shuffles.
__device__ __forceinline__ void tile_logits_fp32(const float* __restrict__ kbase, long long st, int t, int t_end, int D,
                                                 int lane, const float* q_sh, float (&x)[4]) {
  const int g = lane >> 2, c = lane & 3;
  const bool in0 = t + g < t_end, in1 = t + g + 8 < t_end;
  const float* r0 = kbase + (long long)(t + g) * st;
  const float* r1 = r0 + 8 * st;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float s0[kHeads], s1[kHeads];
#pragma unroll
  for (int h = 0; h < kHeads; ++h) s0[h] = s1[h] = 0.f;
  for (int d = 4 * c; d < D; d += 16) {
    const float4 v0 = in0 ? __ldcs(reinterpret_cast<const float4*>(r0 + d)) : zero;
    const float4 v1 = in1 ? __ldcs(reinterpret_cast<const float4*>(r1 + d)) : zero;
#pragma unroll
    for (int h = 0; h < kHeads; ++h) {
      const float4 q = *reinterpret_cast<const float4*>(q_sh + h * kMaxD + d);
      s0[h] = fmaf(v0.w, q.w, fmaf(v0.z, q.z, fmaf(v0.y, q.y, fmaf(v0.x, q.x, s0[h]))));
      s1[h] = fmaf(v1.w, q.w, fmaf(v1.z, q.z, fmaf(v1.y, q.y, fmaf(v1.x, q.x, s1[h]))));
    }
  }
#pragma unroll
  for (int h = 0; h < kHeads; ++h) {
    s0[h] += __shfl_xor_sync(kAll, s0[h], 1); s0[h] += __shfl_xor_sync(kAll, s0[h], 2);
    s1[h] += __shfl_xor_sync(kAll, s1[h], 1); s1[h] += __shfl_xor_sync(kAll, s1[h], 2);
    if (h == 2 * c) { x[0] = s0[h]; x[2] = s1[h]; }
    if (h == 2 * c + 1) { x[1] = s0[h]; x[3] = s1[h]; }
  }
}

// Calls use(first key of the tile, its logits) for every tile of this warp in [lo, hi): tiles warp, warp + kWarps, ..
// While a tile is multiplied the next one's loads are in flight.
template <typename T, int DB, int kWarps, class Use>
__device__ __forceinline__ void for_tiles(const T* __restrict__ kbase, long long st, int lo, int hi, int D, int warp,
                                          int lane, const uint4 (&qr)[DB], const float* q_sh, Use&& use) {
  constexpr int step = kWarps * kRows;
  float x[4];
  int t = lo + warp * kRows;
  if constexpr (sizeof(T) == 4) {
    for (; t < hi; t += step) {
      tile_logits_fp32(kbase, st, t, hi, D, lane, q_sh, x);
      use(t, x);
    }
  } else {
    Tile<DB> p, q;
    if (t < hi) p.load(kbase, st, t, hi, D, lane);
    for (; t < hi; t += 2 * step) {
      if (t + step < hi) q.load(kbase, st, t + step, hi, D, lane);
      p.template logits<T>(qr, x);
      use(t, x);
      if (t + step >= hi) break;
      if (t + 2 * step < hi) p.load(kbase, st, t + 2 * step, hi, D, lane);
      q.template logits<T>(qr, x);
      use(t + step, x);
    }
  }
}

// Grid: one cluster per (layer, sequence, KV head).  DB: 32-channel blocks of a key row.  kStore: the block's logits fit
// in shared memory (cap tokens per head); else (from 51 201 keys on at 8 query heads a pass, 409 601 at one) the second step computes them
// again from K.
template <typename T, int DB, int kWarps, bool kStore>
__global__ void __launch_bounds__(kWarps * 32)
decode_update_kernel(Shape s, TensorView Qn, TensorView K, float scale_log2, float* __restrict__ scores, int cap) {
  extern __shared__ float x_sh[];                                  // [heads of the pass][cap]
  __shared__ alignas(16) float q_sh[sizeof(T) == 4 ? kHeads * kMaxD : 4];   // read as float4
  __shared__ float red[2][kHeads][kWarps];
  __shared__ float part[2][kHeads][2];                             // [pass parity][head]: maximum, sum of this block
  __shared__ float fin[kHeads];                                    // factor of the stored exponentials, or log-sum-exp
  chain_wait();
  chain_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int n_blk = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int unit = blockIdx.x / n_blk;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, c = lane & 3;
  const int hk = unit % s.Hkv;
  const int seq = (unit / s.Hkv) % s.n_seqs;
  const int layer = unit / (s.Hkv * s.n_seqs);
  const int t0 = __ldg(s.cu_seqlens + seq), L = __ldg(s.cu_seqlens + seq + 1) - t0;
  if (L <= 0) return;                                              // uniform over the cluster
  // this block's keys: whole tiles, spread evenly over the cluster
  const int n_tiles = (L + kRows - 1) / kRows, per = (n_tiles + n_blk - 1) / n_blk;
  const int lo = min(L, rank * per * kRows), hi = min(L, lo + per * kRows);
  const T* kbase = static_cast<const T*>(K.ptr) + layer * K.sl + hk * K.sh + (long long)t0 * K.st;
  const float ninf = __int_as_float(0xFF800000);
  // What a logit's exponential is relative to.  Without a maximum all logits are -inf, which adds 0, or NaN, which has to stay.
  auto reference = [&](float maximum) { return maximum == ninf ? 0.f : maximum; };

  int parity = 0;
  for (int g0 = 0; g0 < s.G; g0 += kHeads, parity ^= 1) {          // the group's query heads, 8 at a time
    const int n_heads = min(kHeads, s.G - g0), h0 = hk * s.G + g0;
    const T* q = static_cast<const T*>(Qn.ptr) + layer * Qn.sl + (long long)seq * Qn.st + h0 * Qn.sh;
    uint4 qr[DB];
    if constexpr (sizeof(T) == 2) {
#pragma unroll
      for (int i = 0; i < DB; ++i) {
        const int d = 32 * i + 8 * c;
        qr[i] = g < n_heads && d < s.D ? __ldg(reinterpret_cast<const uint4*>(q + g * Qn.sh + d)) : make_uint4(0u, 0u, 0u, 0u);
      }
    } else {
      __syncthreads();                                             // the previous pass's second step may still read q_sh
      for (int e = tid; e < kHeads * s.D; e += kWarps * 32) {
        const int h = e / s.D, d = e - h * s.D;
        q_sh[h * kMaxD + d] = h < n_heads ? __ldg(reinterpret_cast<const float*>(q + h * Qn.sh) + d) : 0.f;
      }
      __syncthreads();
    }

    // step 1: logits (log2 domain), their maximum and the sum of 2^(x - maximum)
    float mx[2] = {ninf, ninf}, sum[2] = {0.f, 0.f};
    for_tiles<T, DB, kWarps>(kbase, K.st, lo, hi, s.D, warp, lane, qr, q_sh, [&](int t, const float (&x)[4]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = t + g + (i >> 1) * 8, h = 2 * c + (i & 1);
        if (tok < hi && h < n_heads) {
          const float v = x[i] * scale_log2;
          if constexpr (kStore) {
            x_sh[h * cap + tok - lo] = v;
            mx[i & 1] = fmaxf(mx[i & 1], v);
          } else if (v > mx[i & 1]) {
            sum[i & 1] = sum[i & 1] * exp2f(mx[i & 1] - v) + 1.f;
            mx[i & 1] = v;
          } else {
            sum[i & 1] += exp2f(v - reference(mx[i & 1]));
          }
        }
      }
    });
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float big = mx[j];
#pragma unroll
      for (int d = 4; d < 32; d <<= 1) big = fmaxf(big, __shfl_xor_sync(kAll, big, d));
      if constexpr (!kStore) {
        float p = sum[j] == 0.f ? 0.f : sum[j] * exp2f(mx[j] - big);
#pragma unroll
        for (int d = 4; d < 32; d <<= 1) p += __shfl_xor_sync(kAll, p, d);
        if (g == 0) red[1][2 * c + j][warp] = p;
      }
      if (g == 0) red[0][2 * c + j][warp] = big;
    }
    __syncthreads();
    if constexpr (kStore) {
      // sums from shared memory: all threads on one head after the other; the exponentials stay there, so that the
      // second step only scales them
      for (int h = 0; h < n_heads; ++h) {
        float m = ninf;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = fmaxf(m, red[0][h][w]);
        float p = 0.f;
        const float ref = reference(m);
        for (int i = tid; i < hi - lo; i += kWarps * 32) {
          const float e = exp2f(x_sh[h * cap + i] - ref);
          x_sh[h * cap + i] = e;
          p += e;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) p += __shfl_xor_sync(kAll, p, d);
        if (lane == 0) red[1][h][warp] = p;
      }
      __syncthreads();
    }
    if (tid < n_heads) {
      float m = ninf, p = 0.f;
      for (int w = 0; w < kWarps; ++w) m = fmaxf(m, red[0][tid][w]);
      for (int w = 0; w < kWarps; ++w) {
        const float sw = red[1][tid][w];
        p += kStore ? sw : sw == 0.f ? 0.f : sw * exp2f(red[0][tid][w] - m);
      }
      part[parity][tid][0] = m;                                    // -inf: no key, or none with a logit above -inf
      part[parity][tid][1] = p;
    }
    // also keeps a block from rewriting `part` two passes later while a peer still reads it
    if (n_blk > 1) cluster.sync(); else __syncthreads();

    // the group's log-sum-exp: warp = head, lane = block of the cluster
    for (int h = warp; h < n_heads; h += kWarps) {
      float m = ninf, p = 0.f;
      if (lane < n_blk) {
        const float* peer = cluster.map_shared_rank(&part[parity][h][0], lane);
        m = peer[0];
        p = peer[1];
      }
      float all_m = m;
#pragma unroll
      for (int d = 1; d < kMaxCluster; d <<= 1) all_m = fmaxf(all_m, __shfl_xor_sync(kAll, all_m, d));
      p = p == 0.f ? 0.f : p * exp2f(m - all_m);
#pragma unroll
      for (int d = 1; d < kMaxCluster; d <<= 1) p += __shfl_xor_sync(kAll, p, d);
      // stored exponentials are relative to this block's maximum
      if (lane == 0) fin[h] = kStore ? exp2f(part[parity][h][0] - all_m) / p : all_m + log2f(p);
    }
    __syncthreads();

    // step 2: the block's part of the attention row is added.  Every score is owned by one thread, so the result does
    // not depend on the order; the reduction instruction only spares the block the wait for the old values
    // (169 -> 141 us at 32 x 16 x 680 keys, where a block has 24 of them per thread).  It flushes subnormal results, so the
    // smallest weights are added by a load and a store.
    if constexpr (kStore) {
      for (int h = 0; h < n_heads; ++h) {
        float* out = scores + ((long long)layer * s.Hq + h0 + h) * s.T + t0 + lo;
        const float f = fin[h];
        bool tiny = false;
#pragma unroll 4
        for (int i = tid; i < hi - lo; i += kWarps * 32) {
          const float v = x_sh[h * cap + i] * f;
          if (!(v < 0x1p-100f)) atomicAdd(out + i, v);
          tiny |= v < 0x1p-100f && v > 0.f;
        }
        if (tiny)
          for (int i = tid; i < hi - lo; i += kWarps * 32) {
            const float v = x_sh[h * cap + i] * f;
            if (v < 0x1p-100f && v > 0.f) __stcg(out + i, __ldcg(out + i) + v);
          }
      }
    } else {
      for_tiles<T, DB, kWarps>(kbase, K.st, lo, hi, s.D, warp, lane, qr, q_sh, [&](int t, const float (&x)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tok = t + g + (i >> 1) * 8, h = 2 * c + (i & 1);
          if (tok < hi && h < n_heads)
            scores[((long long)layer * s.Hq + h0 + h) * s.T + t0 + tok] += exp2f(x[i] * scale_log2 - fin[h]);
        }
      });
    }
    if (g0 + kHeads < s.G) __syncthreads();                        // x_sh and red are rewritten by the next pass
  }
  if (n_blk > 1) cluster.sync();                                   // peers may still read this block's `part`
}

template <typename T, int DB, int kWarps, bool kStore>
int launch_one(const Shape& s, const TensorView& Qn, const TensorView& K, float scale_log2, float* scores, int n_blk, int cap,
               size_t dyn, cudaStream_t stream) {
  auto kern = decode_update_kernel<T, DB, kWarps, kStore>;
  if (dyn > 32 * 1024 && allow_dynamic_smem(kern, kMaxStored) != KVCRUSH_OK) return KVCRUSH_ERR_CUDA;
  return launch_chained(kern, dim3((unsigned)((long long)s.n_layers * s.n_seqs * s.Hkv * n_blk)), dim3(kWarps * 32), dyn, stream,
                        n_blk, s, Qn, K, scale_log2, scores, cap);
}

template <typename T, int DB>
int launch_width(const Shape& s, const TensorView& Qn, const TensorView& K, float scale_log2, float* scores,
                 cudaStream_t stream) {
  const long long units = (long long)s.n_layers * s.n_seqs * s.Hkv;
  const int n_heads = s.G < kHeads ? s.G : kHeads;
  auto tokens = [&](int n_blk) { return ((s.max_seqlen + kRows - 1) / kRows + n_blk - 1) / n_blk * kRows; };
  auto bytes = [&](int n_blk) { return (size_t)n_heads * tokens(n_blk) * sizeof(float); };
  // Blocks per unit: enough of them for about eight per SM (the last wave is then a small part of the run), none with
  // fewer than 256 keys, and at most 16 KB of logits a block while the cluster can grow.
  const int n_sms = sm_count();
  int n_blk = 1;
  while (n_blk < kMaxCluster && 2 * units * n_blk <= 0x7FFFFFFFLL && tokens(n_blk) > 256 &&
         (units * n_blk < 8 * n_sms || bytes(n_blk) > 16 * 1024))
    n_blk *= 2;
  if (units * n_blk > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  const size_t dyn = bytes(n_blk);
  const int cap = tokens(n_blk);
  // Small blocks, so that while some of an SM's blocks exchange sums and write, the others read: 4 warps 351 us against
  // 358 us with 8 at 32 x 32 x 8192 keys, 169 against 214 us at 32 x 16 x 680 keys.  Where only one or two blocks fit
  // an SM it takes 8 warps to have enough loads in flight.
  if (dyn > kMaxStored) return launch_one<T, DB, 4, false>(s, Qn, K, scale_log2, scores, n_blk, cap, 0, stream);
  if (dyn > 64 * 1024) return launch_one<T, DB, 8, true>(s, Qn, K, scale_log2, scores, n_blk, cap, dyn, stream);
  return launch_one<T, DB, 4, true>(s, Qn, K, scale_log2, scores, n_blk, cap, dyn, stream);
}

template <typename T>
int run_decode(const Shape& s, const TensorView& Qn, const TensorView& K, float scale_log2, float* scores,
               cudaStream_t stream) {
  if constexpr (sizeof(T) == 4) return launch_width<T, 1>(s, Qn, K, scale_log2, scores, stream);
  switch ((s.D + 31) / 32) {
    case 1: return launch_width<T, 1>(s, Qn, K, scale_log2, scores, stream);
    case 2: return launch_width<T, 2>(s, Qn, K, scale_log2, scores, stream);
    case 3: return launch_width<T, 3>(s, Qn, K, scale_log2, scores, stream);
    case 4: return launch_width<T, 4>(s, Qn, K, scale_log2, scores, stream);
    case 5: case 6: return launch_width<T, 6>(s, Qn, K, scale_log2, scores, stream);
    default: return launch_width<T, 8>(s, Qn, K, scale_log2, scores, stream);
  }
}

}  // namespace

int launch_score_decode(const Shape& s, const TensorView& Q_new, const TensorView& K, float scale_log2, float* scores,
                        cudaStream_t stream) {
  if (s.D > kMaxD || s.D % 8 != 0) return KVCRUSH_ERR_UNSUPPORTED;
  if (s.T == 0) return KVCRUSH_OK;
  if (Q_new.dtype == KVCRUSH_FP32) return run_decode<float>(s, Q_new, K, scale_log2, scores, stream);
  if (Q_new.dtype == KVCRUSH_BF16) return run_decode<__nv_bfloat16>(s, Q_new, K, scale_log2, scores, stream);
  if (Q_new.dtype == KVCRUSH_FP16) return run_decode<__half>(s, Q_new, K, scale_log2, scores, stream);
  return KVCRUSH_ERR_UNSUPPORTED;
}

}  // namespace kvc

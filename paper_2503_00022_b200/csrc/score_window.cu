// Stage 1 with an observation window (Sec. 2.3 of the paper: only the last queries of a sequence vote), windows of up to
// 64 queries, on the tensor cores, in one pass over the keys.
//
// Bound by reading K: a window of w queries makes 2 w D flops of every key row, so the two sweeps of score_tc.cu, which
// stream K once each, spent their time on loads.  Here the logits stay in TMEM between the two uses: a cluster of 1 to 8
// CTAs shares one (layer, sequence, query head), each CTA multiplies its key tiles with the window's queries
// (S^T: TMEM lane = key, column = query, one accumulator of w columns per tile, up to 512 columns in all),
//   step 1  puts 2^x in the logit's place, sums it over its keys for every query and exchanges the sums through
//           distributed shared memory,
//   step 2  adds 2^x * 2^-lse2(query) over the queries of every key, from the same accumulators.
// The CTAs live for the whole launch; while step 2 works on one unit the next unit's keys are already on their way, and
// its tiles are multiplied as their accumulators become free, so the loads hardly pause.
// Measured, 32 layers x 32 heads x 8192 tokens of 128 channels (2.1 GB of keys): 16 queries 382 us, 32 queries 481 us, 64
// queries 705 us, where the two sweeps take 1150, 1155 and 1122 us; 1000 tokens, 64 queries 77 against 172 us.  With 64
// queries a cluster of 8 needs all its accumulators for one unit, and the chain load - sum - exchange - add is no longer
// hidden by the next unit's loads.  Taken back: clusters of 16 with two units in TMEM (1056 us, and 1277 us with step 2 one
// unit behind: half the keys a CTA, the same chain of latencies), windows of 128 queries (645 against 562 us at 4096 tokens).
//
// 2^x is taken without a maximum: float32 has the range unless logits are extreme.  32 keys x one column block whose
// logits leave [-100, 100] or hold a NaN keep them, count with their exact maxima in step 1 and take 2^(x - lse2) in step 2.
// So a stored 2^x is finite; a query's sum may be NaN, and is then NaN in every key it votes for, and in no other.  For a
// query whose lse2 is above 126, 2^-lse2 would be flushed to zero: the stored 2^x are multiplied by its square root twice.
// A unit with such a query, or one whose sum is NaN, takes step 2 value by value.
//
// Roles: warp 0 issues TMA loads, warp 1 the tcgen05.mma; warps 2..17 are four epilogue groups of four warps.  All waits
// are bounded as in score_tc.cu; all CTAs of a cluster meet once more before they leave, because peers write into their
// shared memory, and one that gave up then waits for the stores that were on their way to it.
#include <cuda.h>

#include <atomic>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace kvc {

namespace {

using namespace tc;

constexpr int kTile = 128;
constexpr int kCols = 512;                   // TMEM columns
constexpr int kCtrlWarps = 2;
constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (kCtrlWarps + kEpiWarps);
constexpr int kMaxRing = 5;                  // key tiles in flight
constexpr int kMaxSlots = 32;                // accumulators (windows of up to 16 queries)
constexpr int kMaxCluster = 8;
constexpr int kMaxN = 64;
constexpr float kNegInf = -__builtin_huge_valf();

struct WinArgs {
  Shape s;
  float scale_log2;
  float* lse_nat_out;        // optional, voting rows only
  float* scores;
  int normalize;
  int bf16;
  int k_steps;               // 16-channel steps of a dot product
  int n_pad;                 // accumulator columns: the window rounded up to 16, 32 or 64
  int ring;
  int n_units;               // n_layers * n_seqs * Hq
  int min_len, max_len;      // > 0: this launch takes the sequences of min_len to max_len tokens
  int32_t* status;
  int withhold_first_item;   // diagnostic: the producer stops before its first copy, so that every consumer's first wait runs out
};

struct WAux {
  unsigned long long k_full[kMaxRing], k_empty[kMaxRing];
  unsigned long long q_full[2], q_empty[2];
  unsigned long long acc_full[kMaxSlots], acc_empty[kMaxSlots];
  unsigned long long epi_bar, part_full[2], drain;
  uint32_t tmem_base;
  int abort_flag;
  int n_unit;                                           // units whose sums this CTA has received
  int by_value;                                         // 1 + the last unit with a query whose lse2 is above 126 or NaN
  alignas(16) float nlse[kMaxN];                        // minus log2 sum of the window's queries, -inf: no vote
  alignas(16) float factor[kMaxN];                      // 2^nlse
  unsigned char kept[kMaxSlots][4][4];                  // [tile][column block][lane quarter]: logits were kept
  float warp_part[kEpiWarps][32][2];                    // (maximum, sum) of a warp's columns
  float part[2][kMaxCluster][kMaxN];                    // [unit parity][CTA of the cluster][query]: log2 sum, -inf: no key
};
constexpr int kAuxBytes = 26624;
static_assert(sizeof(WAux) <= kAuxBytes, "aux block too large");
constexpr int kSmemTiles = 6;                           // 128-row tiles: ring and two query buffers share them

__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
// Store into a peer's shared memory that counts its 4 bytes on the peer's barrier.
__device__ __forceinline__ void peer_store_async(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
// mbar_wait for a barrier that other CTAs complete
__device__ __forceinline__ bool cluster_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, uint32_t polls) {
  for (uint32_t i = 0; i < polls; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if ((i & 31u) == 31u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
// one poll of a barrier that other CTAs complete
__device__ __forceinline__ bool cluster_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 16 or 32 consecutive columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ldn(uint32_t taddr, uint32_t (&v)[16]) { tmem_ld16(taddr, v); }
__device__ __forceinline__ void tmem_waitn(uint32_t (&v)[16]) { tmem_wait16(v); }
__device__ __forceinline__ void tmem_ldn(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, "
      "%24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]),
        "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]),
        "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_waitn(uint32_t (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                 "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
               :: "memory");
}
// the same columns written (asynchronous: tcgen05.wait::st)
__device__ __forceinline__ void tmem_stn(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_stn(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, "
      "%25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]),
        "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
// NaN if any of the three is
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Sums NC values over the lanes of a warp: lane l is left with the sums of columns l * NC / 32 .. (NC = 16: column l / 2).
template <int NC>
__device__ __forceinline__ float column_sums(float (&v)[NC], int lane) {
#pragma unroll
  for (int n = NC / 2, d = 16; d >= 1; d >>= 1, n >>= 1) {
    if (n >= 1) {
      const bool up = lane & d;
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
        v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, d);
      }
    } else {
      v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], d);
    }
  }
  return v[0];
}

// One (layer, sequence, query head); every role derives it identically.
struct Unit {
  int layer, h, hk, t0, L;
  int nv, q0;                // voting queries: tokens q0 .. q0 + nv - 1 of the sequence
  int tile0, n;              // this CTA's key tiles [tile0, tile0 + n)
  __device__ __forceinline__ Unit(const Shape& s, int u, int rank, int n_cta, bool by_seq) {
    int seq;
    if (by_seq) {                                   // sequences slowest: a launch that leaves some out skips them whole
      h = u % s.Hq; u /= s.Hq;
      hk = h / s.G; layer = u % s.n_layers; seq = u / s.n_layers;
    } else {
      const int g = u % s.G; u /= s.G;
      seq = u % s.n_seqs; u /= s.n_seqs;
      hk = u % s.Hkv; layer = u / s.Hkv;
      h = hk * s.G + g;
    }
    t0 = __ldg(s.cu_seqlens + seq);
    L = __ldg(s.cu_seqlens + seq + 1) - t0;
    nv = min(s.window, L); q0 = L - nv;
    const int tiles = (L + kTile - 1) / kTile, per = (tiles + n_cta - 1) / n_cta;
    tile0 = min(tiles, rank * per);
    n = min(tiles, tile0 + per) - tile0;
  }
};

// NC: columns of one epilogue thread in step 1.  kPolls: polls of every bounded wait.
template <int D, int NC, uint32_t kPolls>
__global__ void __launch_bounds__(kThreads, 1)
score_window_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const WinArgs a) {
  constexpr int kTileBytes = kTile * D * 2, kBlockBytes = kTile * 128;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  WAux* aux = reinterpret_cast<WAux*>(smem + kSmemTiles * kTileBytes);
  volatile int* abort_flag = &aux->abort_flag;
  const uint32_t ring_addr = smem_u32(smem);
  const int ring = a.ring, n_pad = a.n_pad;
  const uint32_t q_bytes = (uint32_t)n_pad * D * 2, q_addr = ring_addr + ring * kTileBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Shape& s = a.s;
  uint32_t rank, n_cta;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n_cta));
  // This cluster's units; every role walks through them in the same way.
  const int unit_step = gridDim.x / n_cta;
  const bool by_seq = a.max_len > 0;
  auto unit_from = [&](int u) {                     // the first at or after u whose sequence is in the launch's range
    while (by_seq && u < a.n_units) {
      const int n_lh = s.n_layers * s.Hq, seq = u / n_lh, len = __ldg(s.cu_seqlens + seq + 1) - __ldg(s.cu_seqlens + seq);
      if (len >= a.min_len && len <= a.max_len) break;
      const int left = (seq + 1) * n_lh - u;        // units of this sequence, skipped in steps of the cluster's stride
      u += (left + unit_step - 1) / unit_step * unit_step;
    }
    return u;
  };

  if (tid == 0) {
    for (int i = 0; i < kMaxRing; ++i) { mbar_init(smem_u32(&aux->k_full[i]), 1); mbar_init(smem_u32(&aux->k_empty[i]), 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&aux->q_full[i]), 1);
      mbar_init(smem_u32(&aux->q_empty[i]), 1);
      mbar_init(smem_u32(&aux->part_full[i]), 1);
    }
    for (int i = 0; i < kMaxSlots; ++i) { mbar_init(smem_u32(&aux->acc_full[i]), 1); mbar_init(smem_u32(&aux->acc_empty[i]), 4); }
    mbar_init(smem_u32(&aux->epi_bar), kEpiWarps);
    mbar_init(smem_u32(&aux->drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < 2; ++i) mbar_expect_tx(smem_u32(&aux->part_full[i]), n_cta * n_pad * 4);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  } else if (warp == 1) {
    tmem_alloc(smem_u32(&aux->tmem_base), kCols);
    tmem_relinquish();
  }
  chain_wait();
  chain_trigger();
  if (tid == 0) aux->n_unit = aux->by_value = 0;
  if (tid == 0) aux->abort_flag = *reinterpret_cast<volatile int32_t*>(a.status) != 0;
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // the peers' barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = aux->tmem_base;
  const bool dead = aux->abort_flag != 0;

  if (dead) {
    // nothing to do
  } else if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    if (lane == 0) {
      int rs = 0, n_q = 0, n_k = 0;
      uint32_t ph = 0;
      bool ok = !a.withhold_first_item;
      for (int u = unit_from(blockIdx.x / n_cta); ok && u < a.n_units; u = unit_from(u + unit_step)) {
        const Unit w(s, u, rank, n_cta, by_seq);
        if (w.n == 0) continue;
        const int qs = n_q & 1;
        ok = mbar_wait(smem_u32(&aux->q_empty[qs]), ((n_q >> 1) & 1) ^ 1, abort_flag, kPolls);
        if (!ok) break;
        mbar_expect_tx(smem_u32(&aux->q_full[qs]), q_bytes);
#pragma unroll
        for (int kb = 0; kb < D / 64; ++kb)
          tma_load_4d(q_addr + qs * q_bytes + kb * n_pad * 128, &map_q, smem_u32(&aux->q_full[qs]), kb * 64, w.t0 + w.q0, w.h, w.layer);
        ++n_q;
        for (int i = 0; i < w.n; ++i) {
          ok = mbar_wait(smem_u32(&aux->k_empty[rs]), ph ^ 1, abort_flag, kPolls);
          if (!ok) break;
          mbar_expect_tx(smem_u32(&aux->k_full[rs]), kTileBytes);
#pragma unroll
          for (int kb = 0; kb < D / 64; ++kb)
            tma_load_4d(ring_addr + rs * kTileBytes + kb * kBlockBytes, &map_k, smem_u32(&aux->k_full[rs]), kb * 64,
                        w.t0 + (w.tile0 + i) * kTile, w.hk, w.layer);
          ++n_k;
          if (++rs == ring) { rs = 0; ph ^= 1; }
        }
      }
      if (*abort_flag) {
        // give the copies in flight a bounded time to land before the CTA's shared memory is released
        for (int q = max(0, n_k - ring); q < n_k; ++q)
          for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(smem_u32(&aux->k_full[q % ring]), (q / ring) & 1); ++i) {}
        for (int q = max(0, n_q - 2); q < n_q; ++q)
          for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(smem_u32(&aux->q_full[q & 1]), (q >> 1) & 1); ++i) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (lane == 0) {
      const uint32_t idesc = make_idesc(kTile, n_pad, a.bf16 != 0);
      int rs = 0, n_q = 0;
      uint32_t ph = 0, used = 0;                    // bit i of used: phase of accumulator i
      bool ok = true;
      for (int u = unit_from(blockIdx.x / n_cta); ok && u < a.n_units; u = unit_from(u + unit_step)) {
        const Unit w(s, u, rank, n_cta, by_seq);
        if (w.n == 0) continue;
        const int qs = n_q & 1;
        ok = mbar_wait(smem_u32(&aux->q_full[qs]), (n_q >> 1) & 1, abort_flag, kPolls);
        for (int i = 0; ok && i < w.n; ++i) {
          ok = mbar_wait(smem_u32(&aux->k_full[rs]), ph, abort_flag, kPolls) &&
               mbar_wait(smem_u32(&aux->acc_empty[i]), ((used >> i) & 1) ^ 1, abort_flag, kPolls);
          if (!ok) break;
          used ^= 1u << i;
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            if (k >= a.k_steps) break;
            umma_bf16(tmem_base + i * n_pad, smem_desc_sw128(ring_addr + rs * kTileBytes + (k >> 2) * kBlockBytes + (k & 3) * 32),
                      smem_desc_sw128(q_addr + qs * q_bytes + (k >> 2) * n_pad * 128 + (k & 3) * 32), idesc, k > 0);
          }
          umma_commit(smem_u32(&aux->acc_full[i]));
          umma_commit(smem_u32(&aux->k_empty[rs]));
          if (++rs == ring) { rs = 0; ph ^= 1; }
        }
        if (!ok) break;
        umma_commit(smem_u32(&aux->q_empty[qs]));
        ++n_q;
      }
      if (*abort_flag) {
        umma_commit(smem_u32(&aux->drain));
        for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(smem_u32(&aux->drain), 0); ++i) {}
      }
    }
  } else {
    // ------------------------------ epilogue groups ------------------------------
    const int ew = warp - kCtrlWarps, gi = ew >> 2, quarter = warp & 3, et = tid - 32 * kCtrlWarps;
    const int r = quarter * 32 + lane;              // TMEM lane: key of the tile
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const float scale = a.scale_log2;
    const f32x2 scale2 = splat2(scale);
    const int n_cb = n_pad / NC, cb = gi & (n_cb - 1);             // step 1: this group's column block ..
    const int tpc = 16 / n_cb;                                     // warps that share a column
    const int j0 = gi / n_cb, j_step = 4 / n_cb;                   // .. and its tiles
    uint32_t used = 0;
    int n_sync = 0, n_unit = 0;
    bool ok = true;
    auto epi_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&aux->epi_bar));
      ok = mbar_wait(smem_u32(&aux->epi_bar), n_sync & 1, abort_flag, kPolls) && ok;
      ++n_sync;
      ok = __all_sync(0xFFFFFFFFu, ok);
    };
    auto wait_acc = [&](int i) {
      ok = mbar_wait(smem_u32(&aux->acc_full[i]), (used >> i) & 1, abort_flag, kPolls) && ok;
      ok = __all_sync(0xFFFFFFFFu, ok);
      tc_fence_after();
      return ok;
    };

    for (int u = unit_from(blockIdx.x / n_cta); u < a.n_units; u = unit_from(u + unit_step)) {
      const Unit w(s, u, rank, n_cta, by_seq);
      if (w.L == 0) continue;
      // first column (query) that key `key` may vote under
      auto first_col = [&](int key) { return key >= w.L ? kMaxN : s.causal ? key - w.q0 : 0; };

      // ---- step 1: 2^x in the logit's place, summed over this warp's keys per query ----
      f32x2 sum2[NC / 2];
#pragma unroll
      for (int i = 0; i < NC / 2; ++i) sum2[i] = 0ull;
      uint32_t kept = 0;                            // tiles of this warp that keep their logits
      int warp_first = kMaxN;                       // first column with a key of this warp
      for (int j = j0; j < w.n; j += j_step) {
        if (!wait_acc(j)) break;
        const uint32_t t_acc = t_lane + j * n_pad + cb * NC;
        uint32_t v[NC];
        tmem_ldn(t_acc, v);
        const int key_first = first_col((w.tile0 + j) * kTile + r), c_first = key_first - cb * NC;
        warp_first = min(warp_first, __reduce_min_sync(0xFFFFFFFFu, key_first));
        tmem_waitn(v);
        float hi = 0.f, lo = 0.f;
#pragma unroll
        for (int i = 0; i < NC; i += 2) {
          hi = max3_nan(hi, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
          lo = min3(lo, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
        }
        const bool keep = __any_sync(0xFFFFFFFFu, !(hi * scale < 100.f && lo * scale > -100.f));
        if (lane == 0) aux->kept[j][cb][quarter] = keep;
        if (keep) { kept |= 1u << j; continue; }
        auto exps = [&](auto mixed) {
#pragma unroll
          for (int i = 0; i < NC / 2; ++i) {
            const f32x2 x = mul2(pack2(v[2 * i], v[2 * i + 1]), scale2);
            const f32x2 e = decltype(mixed)::value && (i & 3) == 3 ? exp2_poly2(x) : exp2_sfu2(x);
            sum2[i] = add2(sum2[i], e);
            float e0, e1;
            unpack2(e, e0, e1);
            v[2 * i] = __float_as_uint(e0);
            v[2 * i + 1] = __float_as_uint(e1);
          }
        };
        if (__any_sync(0xFFFFFFFFu, c_first > 0)) {
#pragma unroll
          for (int i = 0; i < NC; ++i) v[i] = i >= c_first ? v[i] : 0xFF800000u;
          exps(std::false_type{});                  // no vote: exactly 2^-inf = 0
        } else {
          exps(std::true_type{});
        }
        tmem_stn(t_acc, v);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      if (!ok) break;
      float v[NC];
#pragma unroll
      for (int i = 0; i < NC / 2; ++i) unpack2(sum2[i], v[2 * i], v[2 * i + 1]);
      const float sum = column_sums<NC>(v, lane);
      const int my_col = NC == 32 ? lane : lane >> 1;
      const bool has_keys = cb * NC + my_col >= warp_first && sum > 0.f;
      if (NC == 32 || (lane & 1) == 0) {
        aux->warp_part[ew][my_col][0] = has_keys ? 0.f : kNegInf;
        aux->warp_part[ew][my_col][1] = has_keys ? sum : 0.f;
      }
      if (kept) {                                   // add the kept tiles, column by column with exact maxima
        __syncwarp();
#pragma unroll 1
        for (int c = 0; c < NC; ++c) {
          float m = aux->warp_part[ew][c][0], t = 0.f;
          const float m0 = m, t0 = aux->warp_part[ew][c][1];
          for (int step = 0; step < 2; ++step) {
            for (int j = j0; j < w.n; j += j_step) {
              if (!((kept >> j) & 1u)) continue;
              uint32_t x;
              asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(x) : "r"(t_lane + j * n_pad + cb * NC + c) : "memory");
              asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(x) :: "memory");
              const bool in = cb * NC + c >= first_col((w.tile0 + j) * kTile + r);
              const float xs = in ? __uint_as_float(x) * scale : kNegInf;
              if (step == 0) m = fmaxf(m, xs);
              else t += ex2(xs - (m == kNegInf ? 0.f : m));            // -inf adds 0, NaN stays
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
              if (step == 0) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
              else t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
            }
          }
          if (m0 != kNegInf) t += t0 * ex2(m0 - m);
          if (lane == 0) { aux->warp_part[ew][c][0] = m; aux->warp_part[ew][c][1] = t; }
          __syncwarp();
        }
      }
      tc_fence_before();
      epi_sync();
      if (!ok) break;

      // ---- the CTA's sums to every CTA of the cluster, then the row log-sum-exp ----
      // Threads (column, i): i stands first for one of the 16 / n_cb warps that summed the column, then for a CTA.
      const int par = n_unit & 1, col = et / tpc, sub = et & (tpc - 1);
      if (col < n_pad) {                            // uniform over a warp
        const int cw = 4 * (col / NC + n_cb * (sub >> 2)) + (sub & 3), ci = col & (NC - 1);
        const float mw = aux->warp_part[cw][ci][0], tw = aux->warp_part[cw][ci][1];
        float m = mw;
        for (int d = 1; d < tpc; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
        float t = tw == 0.f ? 0.f : tw * ex2(mw - m);
        for (int d = 1; d < tpc; d <<= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
        const float l = t == 0.f ? kNegInf : m + log2f(t);
        if (n_cta == 1) {                           // alone: this warp reads it back itself (and a launch without
          if (sub == 0) aux->part[par][0][col] = l; // clusters has no st.async)
          __syncwarp();
        } else {
          for (int p = sub; p < (int)n_cta; p += tpc)
            peer_store_async(peer_addr(smem_u32(&aux->part[par][rank][col]), p), l, peer_addr(smem_u32(&aux->part_full[par]), p));
        }
      }
      if (n_cta > 1) {
        ok = cluster_wait(smem_u32(&aux->part_full[par]), (n_unit >> 1) & 1, abort_flag, kPolls) && ok;
        ok = __all_sync(0xFFFFFFFFu, ok);
      }
      if (col < n_pad) {
        float m = kNegInf, t = 0.f;
        for (int p = sub; p < (int)n_cta; p += tpc) m = fmaxf(m, aux->part[par][p][col]);
        for (int d = 1; d < tpc; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
        for (int p = sub; p < (int)n_cta; p += tpc) t += ex2(aux->part[par][p][col] - m);      // -inf: adds nothing
        for (int d = 1; d < tpc; d <<= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
        if (sub == 0) {
          const float lse2 = m + log2f(t);
          aux->nlse[col] = col < w.nv ? -lse2 : kNegInf;
          if (col < w.nv && !(lse2 <= 126.f)) aux->by_value = n_unit + 1;
          aux->factor[col] = col < w.nv ? ex2(lse2 < -126.f ? 126.f : -lse2) : 0.f;    // beyond 2^126 no column is below 2^100
          if (rank == 0 && col < w.nv && a.lse_nat_out)
            a.lse_nat_out[((size_t)w.layer * s.Hq + w.h) * s.T + w.t0 + w.q0 + col] = lse2 * 0.69314718055994530942f;
        }
      }
      epi_sync();
      if (!ok) break;
      // armed again for the unit after the next: a peer sends that only when it has this CTA's sums of the next unit
      if (et == 0 && n_cta > 1) mbar_expect_tx(smem_u32(&aux->part_full[par]), n_cta * n_pad * 4);

      // ---- step 2: every key's sum over the queries ----
      tc_fence_after();
      const bool by_value = aux->by_value == n_unit + 1;
      for (int j = gi; j < w.n; j += 4) {
        const int key = (w.tile0 + j) * kTile + r;
        const uint32_t t_acc = t_lane + j * n_pad;
        f32x2 acc[2] = {0ull, 0ull};
        for (int b = 0; b < n_cb; ++b) {
          uint32_t x[NC];
          tmem_ldn(t_acc + b * NC, x);
          tmem_waitn(x);
          if (!by_value && !aux->kept[j][b][quarter]) {
            const float4* f4 = reinterpret_cast<const float4*>(aux->factor + b * NC);
#pragma unroll
            for (int i = 0; i < NC / 4; ++i) {
              const float4 f = f4[i];
              acc[0] = fma2(pack2(x[4 * i], x[4 * i + 1]), pack2f(f.x, f.y), acc[0]);
              acc[1] = fma2(pack2(x[4 * i + 2], x[4 * i + 3]), pack2f(f.z, f.w), acc[1]);
            }
          } else {
            const int c_first = first_col(key) - b * NC;
            const bool keep = aux->kept[j][b][quarter];
            float t = 0.f;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
              const float x_i = __uint_as_float(x[i]), nl = aux->nlse[b * NC + i];
              float e;
              if (keep) e = ex2(fmaf(x_i, scale, nl));
              else if (nl < -126.f) { const float root = ex2(0.5f * nl); e = x_i * root * root; }
              else e = x_i * aux->factor[b * NC + i];
              t += i >= c_first ? e : 0.f;
            }
            acc[0] = add2(acc[0], pack2f(t, 0.f));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&aux->acc_empty[j]));
        if (key < w.L) {
          const float total = sum4(acc);
          a.scores[((size_t)w.layer * s.Hq + w.h) * s.T + w.t0 + key] = a.normalize ? total / (float)w.nv : total;
        }
      }
      if (!ok) break;
      if (w.n > 0) used ^= 0xFFFFFFFFu >> (32 - w.n);
      ++n_unit;
    }
    if (et == 0) aux->n_unit = n_unit;
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // nobody leaves while a peer may still write into its shared memory
  if (tid == 0 && n_cta > 1 && *abort_flag) {
    // The barrier does not order the peers' asynchronous stores.  After it none of them sends any more, and what they have
    // sent belongs to the unit this CTA gave up in or the next: a bounded time for it to land.  (A CTA that did not give
    // up has received everything that is sent to it.)
    for (int u = aux->n_unit; u < aux->n_unit + 2; ++u)
      for (uint32_t i = 0; i < kDrainPolls && !cluster_test(smem_u32(&aux->part_full[u & 1]), (u >> 1) & 1); ++i) {}
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kCols);
  }
  if (tid == 0 && !dead && *abort_flag) report(a.status, KVCRUSH_DEV_TIMEOUT, KID_SCORE_WINDOW, blockIdx.x, 0);
}

constexpr int kMaxDevices = 64;

// Clusters of n_cta blocks that run at the same time (write-once cache per device: the answer depends on nothing else).
template <int D, int NC, uint32_t kPolls>
int resident_clusters(int log_cta, int smem) {
  static std::atomic<int> known[kMaxDevices][4];
  auto kern = score_window_kernel<D, NC, kPolls>;
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  if ((n = known[dev][log_cta].load(std::memory_order_relaxed)) > 0) return n;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1u << log_cta);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << log_cta; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  known[dev][log_cta].store(n, std::memory_order_relaxed);
  return n;
}

template <int D, int NC, uint32_t kPolls>
int launch_window_polls(const CUtensorMap& mq, const CUtensorMap& mk, const WinArgs& a, int units, int log_cta, cudaStream_t stream) {
  constexpr int smem = kSmemTiles * kTile * D * 2 + kAuxBytes + 1024;
  auto kern = score_window_kernel<D, NC, kPolls>;
  const int clusters = resident_clusters<D, NC, kPolls>(log_cta, smem);
  if (clusters < 1) return KVCRUSH_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return KVCRUSH_ERR_CUDA;
  const int n = clusters < units ? clusters : units;
  return launch_chained(kern, dim3((unsigned)n << log_cta), dim3(kThreads), smem, stream, 1 << log_cta, mq, mk, a);
}

template <int D, int NC>
int launch_window(const CUtensorMap& mq, const CUtensorMap& mk, const WinArgs& a, int units, int log_cta, bool short_waits,
                  cudaStream_t stream) {
  return short_waits ? launch_window_polls<D, NC, kShortWaitPolls>(mq, mk, a, units, log_cta, stream)
                     : launch_window_polls<D, NC, kWaitPolls>(mq, mk, a, units, log_cta, stream);
}

int pad_window(int window) {
  int n_pad = 16;
  while (n_pad < window) n_pad *= 2;
  return n_pad;
}

// CTAs per cluster: as few as hold the logits, more while the launch would leave SMs idle.  A batch whose sequences need
// clusters of different sizes is launched once for each size, longest first, if that spares at least two rounds of the
// chip: 8192 and 15 x 300 tokens (4 layers x 32 heads, 64 queries) 744 -> 198 us (the two sweeps 348), 4200 and 4000 tokens
// (1 layer) 45 us together, 47 apart.
struct Plan {
  int cta_tokens;            // keys whose logits one CTA holds
  long long units[4], together;      // (layer, sequence, head)s by the log2 of the cluster size they need, and all of them
  int longest[4], largest;   // longest sequence of a size, largest size
  bool split;
};
Plan plan_launches(const Shape& s, const int32_t* cu_host, int n_sms, int n_pad) {
  Plan p{};
  p.cta_tokens = kCols / n_pad * kTile;
  for (int i = 0; i < s.n_seqs; ++i) {
    const int len = cu_host[i + 1] - cu_host[i];
    if (len == 0) continue;
    int need = 0;
    while (len > p.cta_tokens << need) ++need;
    p.units[need] += (long long)s.n_layers * s.Hq;
    p.longest[need] = len > p.longest[need] ? len : p.longest[need];
    p.largest = need > p.largest ? need : p.largest;
  }
  auto rounds = [&](long long n, int log_cta) {
    const int clusters = n_sms >> log_cta > 0 ? n_sms >> log_cta : 1;
    return (n + clusters - 1) / clusters;
  };
  long long apart = 0;
  for (int need = 0; need < 4; ++need) { apart += rounds(p.units[need], need); p.together += p.units[need]; }
  p.split = rounds(p.together, p.largest) >= apart + 2;
  return p;
}

}  // namespace

// The one-pass kernel takes windows of up to 64 queries when the logits of a cluster's keys fit its TMEM: sequences of
// up to 65536 / (window rounded up) x 8 tokens; the rest goes to the two sweeps.
bool score_window_fits(const Shape& s) {
  if (s.window < 1 || s.window > kMaxN || s.max_seqlen < 1) return false;
  const int tiles = (s.max_seqlen + kTile - 1) / kTile;
  return (tiles + kMaxCluster - 1) / kMaxCluster * pad_window(s.window) <= kCols && (long long)s.n_layers * s.n_seqs * s.Hq <= 0x7FFFFFFFLL / kMaxCluster;
}

int score_window_launches(const Shape& s, const int32_t* cu_host) {
  const Plan p = plan_launches(s, cu_host, sm_count(), pad_window(s.window));
  int n = 0;
  for (int need = 0; need < 4; ++need) n += p.units[need] > 0;
  return p.split ? n : 1;
}

int launch_score_window(const Shape& s, const int32_t* cu_host, const TensorView& Q, const ScoreTensorMaps& maps, float scale_log2, float* scores,
                        float* lse_out, int normalize, int32_t* status, const ScoreDiag& diag, cudaStream_t stream) {
  WinArgs a{};
  a.s = s; a.scale_log2 = scale_log2; a.lse_nat_out = lse_out; a.scores = scores; a.normalize = normalize;
  a.bf16 = Q.dtype == KVCRUSH_BF16; a.status = status; a.k_steps = (s.D + 15) / 16;
  a.withhold_first_item = diag.withhold_first_item;
  a.n_units = s.n_layers * s.n_seqs * s.Hq;
  a.n_pad = pad_window(s.window);
  a.ring = kMaxRing;                                // two query buffers of n_pad rows take the sixth tile at most
  CUtensorMap mq;
  if (!make_map(&mq, Q, s.D, s.T, s.Hq, s.n_layers, a.n_pad)) return KVCRUSH_ERR_UNSUPPORTED;
  const CUtensorMap& mk = *reinterpret_cast<const CUtensorMap*>(maps.k);
  const bool sw = diag.short_waits != 0;
  auto launch = s.D > 64 ? (a.n_pad == 16 ? launch_window<128, 16> : launch_window<128, 32>)
                         : (a.n_pad == 16 ? launch_window<64, 16> : launch_window<64, 32>);
  const int n_sms = sm_count();
  const Plan plan = plan_launches(s, cu_host, n_sms, a.n_pad);
  for (int need = plan.largest; need >= 0; --need) {
    const long long n = plan.split ? plan.units[need] : plan.together;
    if (n == 0) continue;
    if (plan.split) {
      a.min_len = need == 0 ? 1 : (plan.cta_tokens << (need - 1)) + 1;
      a.max_len = plan.cta_tokens << need;
    }
    const int tiles = (plan.longest[need] + kTile - 1) / kTile;
    int log_cta = need;
    while (log_cta < 3 && (tiles + (1 << log_cta) - 1) >> log_cta > 1 && n << (log_cta + 1) <= n_sms) ++log_cta;
    const int rc = launch(mq, mk, a, (int)n, log_cta, sw, stream);
    if (rc != KVCRUSH_OK || !plan.split) return rc;
  }
  return KVCRUSH_OK;
}

}  // namespace kvc

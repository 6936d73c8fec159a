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
// The CTAs live for the whole launch.  Sixteen warps do step 1, four others the exchange and step 2; they hand units on through
// barriers, and unit after unit takes the next accumulators round and round, so that loads, products, exponentials and sums of
// up to three units overlap.  (With all warps at one unit's steps in turn the chain exponentials - exchange - sums was the
// time.)  For a launch's last unit all of them share step 2.
// Measured, 32 layers x 32 heads x 8192 tokens of 128 channels (2.1 GB of keys): 16 queries 354 us, 32 queries 434 us, 64
// queries 596 us (with one group of warps for all steps 375, 512, 732; the two sweeps 1150, 1155 and 1122); 1000 tokens, 64
// queries 68.6 us (79.6; 172), 8 layers of 5003 + 3117 tokens 176 (238), 8 layers x 40 heads of 12000 tokens, 32 queries 223 (293).
// With 64 queries a cluster of 8 needs all its accumulators for one unit, and step 1 of the next one follows step 2 tile by
// tile.  Taken back: clusters of 16 with two units in TMEM (1056 us, and 1277 with step 2 one unit behind: half the keys a CTA,
// the same chain of latencies), windows of 128 queries (645 against 562 us at 4096 tokens, with one group of warps).
//
// 2^x is taken without a maximum: float32 has the range unless logits are extreme.  32 keys x one column block whose
// logits leave [-100, 100] or hold a NaN keep them, count with their exact maxima in step 1 and take 2^(x - lse2) in step 2.
// So a stored 2^x is finite; a query's sum may be NaN, and is then NaN in every key it votes for, and in no other.  For a
// query whose lse2 is above 126, 2^-lse2 would be flushed to zero: the stored 2^x are multiplied by its square root twice.
// A unit with such a query, with one whose sum is NaN, or with kept logits takes step 2 value by value, with one decision for
// 16 values (a branch for each made one kept block cost a unit ten times its step 2).  8 layers x 32 heads x 8192 tokens, 64
// queries, four keys with logits of 75: 1021 -> 473 us (with one group of warps for all steps 540), one in 128 keys 1277 -> 743
// (760), all queries times 60: 981 -> 755 (768), logits of 95 959 -> 480 (625); the rest is step 1's sums with exact maxima.
//
// Roles: warp 0 issues TMA loads, warp 1 the tcgen05.mma; warps 4..7 are the group of the exchange and step 2, warps 8..23 the
// four groups of step 1.  (Step 2, on which the accumulators wait, before step 1 in the order of the warps, and without copies
// between its two buffers: 64 queries of 8192 tokens 632 -> 606 us, of 4096 292 -> 280; 32 queries of 8192 431 -> 434.)  All waits
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
constexpr int kCtrlWarps = 4;                // one warpgroup: producer, issuer, two idle warps
constexpr int kExpWarps = 16;                // four groups of four: step 1
constexpr int kSumWarps = 4;                 // one group: exchange and step 2
constexpr int kThreads = 32 * (kCtrlWarps + kExpWarps + kSumWarps);
constexpr int kNC = 16;                      // columns of a step-1 thread
// Registers: 80 a thread at launch (the most 24 warps can have); the control warpgroup gives some to the group of step 2.  With
// 48 and 112 the producer and the issuer spill: 714 us instead of 633 for 64 queries of 8192 tokens.
constexpr int kLaunchRegs = 80, kCtrlRegs = 64, kSumRegs = 96;
static_assert(32 * (kCtrlWarps * kCtrlRegs + kExpWarps * kLaunchRegs + kSumWarps * kSumRegs) <= kThreads * kLaunchRegs,
              "register split within the launch's total");
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
  unsigned long long sums_full[2], sums_empty[2];       // [unit parity]: warp_part and kept
  unsigned long long sum_bar, part_full[2], last_unit, drain;
  uint32_t tmem_base;
  int abort_flag;
  int n_unit;                                           // units whose sums this CTA has received
  int any_kept[2];                                      // [unit parity] 1 + the last unit that kept logits
  int last_by_value;                                    // the last unit's step 2 goes value by value
  alignas(16) float nlse[kSumWarps][kMaxN];             // [warp of step 2] minus log2 sum of the window's queries, -inf: no vote
  alignas(16) float factor[kSumWarps][kMaxN];           // 2^nlse, or its root if that is below the normal numbers ..
  alignas(16) float factor2[kSumWarps][kMaxN];          // .. and then the root again, else 1
  uint32_t kept[2][kExpWarps];                          // [unit parity] tiles (bits) whose logits a warp of step 1 kept
  float warp_part[2][kExpWarps][kNC][2];                // [unit parity] (maximum, sum) of a warp's columns
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

// 16 columns written (asynchronous: tcgen05.wait::st)
__device__ __forceinline__ void tmem_stn(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
// the largest magnitude, NaN if any of the three is
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(fabsf(b)), "f"(fabsf(c)));
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

// NP: accumulator columns, the window rounded up to 16, 32 or 64.  kPolls: polls of every bounded wait.
template <int D, int NP, uint32_t kPolls>
__global__ void __launch_bounds__(kThreads, 1)
score_window_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const WinArgs a) {
  constexpr int kSlots = kCols / NP;                // accumulators; unit after unit takes the next ones, round and round
  constexpr int kTileBytes = kTile * D * 2, kBlockBytes = kTile * 128;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  WAux* aux = reinterpret_cast<WAux*>(smem + kSmemTiles * kTileBytes);
  volatile int* abort_flag = &aux->abort_flag;
  const uint32_t ring_addr = smem_u32(smem);
  const int ring = a.ring;
  constexpr uint32_t q_bytes = NP * D * 2;
  const uint32_t q_addr = ring_addr + ring * kTileBytes;
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
      mbar_init(smem_u32(&aux->sums_full[i]), kExpWarps);
      mbar_init(smem_u32(&aux->sums_empty[i]), kSumWarps);
    }
    for (int i = 0; i < kMaxSlots; ++i) { mbar_init(smem_u32(&aux->acc_full[i]), 1); mbar_init(smem_u32(&aux->acc_empty[i]), kSumWarps); }
    mbar_init(smem_u32(&aux->sum_bar), kSumWarps);
    mbar_init(smem_u32(&aux->last_unit), kSumWarps);
    mbar_init(smem_u32(&aux->drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < 2; ++i) mbar_expect_tx(smem_u32(&aux->part_full[i]), n_cta * NP * 4);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  } else if (warp == 1) {
    tmem_alloc(smem_u32(&aux->tmem_base), kCols);
    tmem_relinquish();
  }
  chain_wait();
  chain_trigger();
  if (tid == 0) aux->n_unit = aux->any_kept[0] = aux->any_kept[1] = aux->last_by_value = 0;
  if (tid == 0) aux->abort_flag = *reinterpret_cast<volatile int32_t*>(a.status) != 0;
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // the peers' barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = aux->tmem_base;
  const bool dead = aux->abort_flag != 0;

  if (dead) {
    // nothing to do
  } else if (warp < kCtrlWarps) {
  set_max_regs<kCtrlRegs, false>();
  if (warp == 0) {
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
          tma_load_4d(q_addr + qs * q_bytes + kb * NP * 128, &map_q, smem_u32(&aux->q_full[qs]), kb * 64, w.t0 + w.q0, w.h, w.layer);
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
      const uint32_t idesc = make_idesc(kTile, NP, a.bf16 != 0);
      int rs = 0, n_q = 0;
      uint32_t ph = 0, n_acc = 0;                   // accumulators handed out
      bool ok = true;
      for (int u = unit_from(blockIdx.x / n_cta); ok && u < a.n_units; u = unit_from(u + unit_step)) {
        const Unit w(s, u, rank, n_cta, by_seq);
        if (w.n == 0) continue;
        const int qs = n_q & 1;
        ok = mbar_wait(smem_u32(&aux->q_full[qs]), (n_q >> 1) & 1, abort_flag, kPolls);
        for (int i = 0; ok && i < w.n; ++i, ++n_acc) {
          const int slot = n_acc & (kSlots - 1);
          ok = mbar_wait(smem_u32(&aux->k_full[rs]), ph, abort_flag, kPolls) &&
               mbar_wait(smem_u32(&aux->acc_empty[slot]), (n_acc / kSlots & 1) ^ 1, abort_flag, kPolls);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            if (k >= a.k_steps) break;
            umma_bf16(tmem_base + slot * NP, smem_desc_sw128(ring_addr + rs * kTileBytes + (k >> 2) * kBlockBytes + (k & 3) * 32),
                      smem_desc_sw128(q_addr + qs * q_bytes + (k >> 2) * NP * 128 + (k & 3) * 32), idesc, k > 0);
          }
          umma_commit(smem_u32(&aux->acc_full[slot]));
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
  }
  } else {
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;              // TMEM lane: key of the tile
    const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const float scale = a.scale_log2;
    constexpr int n_cb = NP / kNC, j_step = 4 / n_cb;   // column blocks of step 1, and groups that share one
    uint32_t n_acc = 0;                             // accumulators taken by earlier units
    int n_unit = 0;
    bool ok = true;
    auto slot_of = [&](int j) { return (int)((n_acc + j) & (kSlots - 1)); };
    auto wait_for = [&](unsigned long long& bar, uint32_t parity) {
      ok = mbar_wait(smem_u32(&bar), parity, abort_flag, kPolls) && ok;
      ok = __all_sync(0xFFFFFFFFu, ok);
      return ok;
    };

    auto store = [&](const Unit& w, int j, float total) {
      const int key = (w.tile0 + j) * kTile + r;
      if (key < w.L) a.scores[((size_t)w.layer * s.Hq + w.h) * s.T + w.t0 + key] = a.normalize ? total / (float)w.nv : total;
    };
    // Step 2 of one tile, value by value: logits were kept in the unit, or a query's 2^-lse2 is not a normal number (or NaN).
    auto by_value_tile = [&](const Unit& w, int j, int par, int copy) {
      const int slot = slot_of(j), key = (w.tile0 + j) * kTile + r;
      const int c_first = key >= w.L ? kMaxN : s.causal ? key - w.q0 : 0;
      float total[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int b = 0; b < n_cb; ++b) {
        uint32_t x[kNC];
        tmem_ld16(t_lane + slot * NP + b * kNC, x);
        tmem_wait16(x);
        const bool keep = aux->kept[par][4 * (b + n_cb * (j & (j_step - 1))) + quarter] >> j & 1u;
        const int first = c_first - b * kNC;
        if (keep) {
#pragma unroll
          for (int i = 0; i < kNC; i += 4) {
            const float4 n4 = *reinterpret_cast<const float4*>(&aux->nlse[copy][b * kNC + i]);
            const float nl[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {           // -inf: no voting query, whatever the logit is (inf and NaN included)
              const float e = ex2(fmaf(__uint_as_float(x[i + k]), scale, nl[k]));
              total[k] += i + k >= first && nl[k] != kNegInf ? e : 0.f;
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < kNC; i += 4) {
            const float4 f4 = *reinterpret_cast<const float4*>(&aux->factor[copy][b * kNC + i]);
            const float4 g4 = *reinterpret_cast<const float4*>(&aux->factor2[copy][b * kNC + i]);
            const float f[4] = {f4.x, f4.y, f4.z, f4.w}, g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float e = __uint_as_float(x[i + k]) * f[k] * g[k];
              total[k] += i + k >= first ? e : 0.f;
            }
          }
        }
      }
      return (total[0] + total[1]) + (total[2] + total[3]);
    };

    if (warp >= kCtrlWarps + kSumWarps) {
      // ------------------------------ step 1: 2^x in the logit's place, summed over this warp's keys per query ------
      const int ew = warp - kCtrlWarps - kSumWarps, gi = ew >> 2;
      const f32x2 scale2 = splat2(scale);
      const int cb = gi & (n_cb - 1), j0 = gi / n_cb;   // this group's column block and first tile
      for (int u = unit_from(blockIdx.x / n_cta); u < a.n_units; u = unit_from(u + unit_step)) {
        const Unit w(s, u, rank, n_cta, by_seq);
        if (w.L == 0) continue;
        const int par = n_unit & 1;
        const int key_end = s.causal ? min(w.L, w.q0 + cb * kNC + 1) : w.L;   // keys below vote under every column of the block
        // first column (query) that key `key` may vote under
        auto first_col = [&](int key) { return key >= w.L ? kMaxN : s.causal ? key - w.q0 : 0; };
        f32x2 sum2[kNC / 2];
#pragma unroll
        for (int i = 0; i < kNC / 2; ++i) sum2[i] = 0ull;
        uint32_t kept = 0;                          // tiles of this warp that keep their logits
        for (int j = j0; j < w.n; j += j_step) {
          const int slot = slot_of(j);
          if (!wait_for(aux->acc_full[slot], (n_acc + j) / kSlots & 1)) break;
          tc_fence_after();
          const uint32_t t_acc = t_lane + slot * NP + cb * kNC;
          uint32_t v[kNC];
          tmem_ld16(t_acc, v);
          tmem_wait16(v);
          float hi = 0.f;
#pragma unroll
          for (int i = 0; i < kNC; i += 2) hi = max3_abs(hi, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
          if (__any_sync(0xFFFFFFFFu, !(hi * scale < 100.f))) { kept |= 1u << j; continue; }
          auto exps = [&](auto mixed) {
#pragma unroll
            for (int i = 0; i < kNC / 2; ++i) {
              const f32x2 x = mul2(pack2(v[2 * i], v[2 * i + 1]), scale2);
              const f32x2 e = decltype(mixed)::value && (i & 3) == 3 ? exp2_poly2(x) : exp2_sfu2(x);
              sum2[i] = add2(sum2[i], e);
              float e0, e1;
              unpack2(e, e0, e1);
              v[2 * i] = __float_as_uint(e0);
              v[2 * i + 1] = __float_as_uint(e1);
            }
          };
          const int tile_key = (w.tile0 + j) * kTile;
          if (tile_key + kTile > key_end) {         // uniform over the group
            const int c_first = first_col(tile_key + r) - cb * kNC;
#pragma unroll
            for (int i = 0; i < kNC; ++i) v[i] = i >= c_first ? v[i] : 0xFF800000u;
            exps(std::false_type{});                // no vote: exactly 2^-inf = 0
          } else {
            exps(std::true_type{});
          }
          tmem_stn(t_acc, v);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        if (!ok) break;
        float v[kNC];
#pragma unroll
        for (int i = 0; i < kNC / 2; ++i) unpack2(sum2[i], v[2 * i], v[2 * i + 1]);
        const float sum = column_sums<kNC>(v, lane);
        if (!wait_for(aux->sums_empty[par], (n_unit >> 1 & 1) ^ 1)) break;
        float (*part)[2] = aux->warp_part[par][ew];
        if ((lane & 1) == 0) {
          part[lane >> 1][0] = sum > 0.f ? 0.f : kNegInf;
          part[lane >> 1][1] = sum;
        }
        if (lane == 0) aux->kept[par][ew] = kept;
        if (kept) {                                 // add the kept tiles, column by column with exact maxima
          if (lane == 0) aux->any_kept[par] = n_unit + 1;
          __syncwarp();
#pragma unroll 1
          for (int c = 0; c < kNC; ++c) {
            float m = part[c][0], t = 0.f;
            const float m0 = m, t0 = part[c][1];
            for (int step = 0; step < 2; ++step) {
              for (int j = j0; j < w.n; j += j_step) {
                if (!((kept >> j) & 1u)) continue;
                uint32_t x;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];"
                             : "=r"(x) : "r"(t_lane + slot_of(j) * NP + cb * kNC + c) : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(x) :: "memory");
                const bool in = cb * kNC + c >= first_col((w.tile0 + j) * kTile + r);
                const float xs = in ? __uint_as_float(x) * scale : kNegInf;
                if (step == 0) m = fmaxf(m, xs);
                else t += ex2(xs - (m == kNegInf ? 0.f : m));          // -inf adds 0, NaN stays
              }
#pragma unroll
              for (int d = 16; d > 0; d >>= 1) {
                if (step == 0) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
                else t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
              }
            }
            if (m0 != kNegInf) t += t0 * ex2(m0 - m);
            __syncwarp();
            if (lane == 0) { part[c][0] = m; part[c][1] = t; }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&aux->sums_full[par]));
        if (unit_from(u + unit_step) >= a.n_units) {    // the last unit: nothing else to do than to share its step 2
          if (!wait_for(aux->last_unit, 0)) break;
          tc_fence_after();
          const bool by_value = aux->last_by_value != 0;
          for (int j = 1 + gi; j < w.n; j += 5) {
            f32x2 acc[2] = {0ull, 0ull};
            if (!by_value) {
#pragma unroll
              for (int b = 0; b < n_cb; ++b) {
                uint32_t x[kNC];
                tmem_ld16(t_lane + slot_of(j) * NP + b * kNC, x);
                tmem_wait16(x);
                const float4* f4 = reinterpret_cast<const float4*>(aux->factor[0] + b * kNC);
#pragma unroll
                for (int i = 0; i < kNC / 4; ++i) {
                  const float4 f = f4[i];
                  acc[0] = fma2(pack2(x[4 * i], x[4 * i + 1]), pack2f(f.x, f.y), acc[0]);
                  acc[1] = fma2(pack2(x[4 * i + 2], x[4 * i + 3]), pack2f(f.z, f.w), acc[1]);
                }
              }
            }
            store(w, j, by_value ? by_value_tile(w, j, par, 0) : sum4(acc));
          }
        }
        n_acc += w.n;
        ++n_unit;
      }
    } else {
      // ------------------------------ exchange, then step 2: every key's sum over the queries -----------------------
      set_max_regs<kSumRegs, true>();
      const int st = tid - 32 * kCtrlWarps;
      constexpr int tpc = 32 * kSumWarps / NP;      // threads of a column: i stands first for warps that summed it, then for CTAs
      const int col = st / tpc, sub = st & (tpc - 1);
      for (int u = unit_from(blockIdx.x / n_cta); u < a.n_units; u = unit_from(u + unit_step)) {
        const Unit w(s, u, rank, n_cta, by_seq);
        if (w.L == 0) continue;
        const int par = n_unit & 1;
        if (!wait_for(aux->sums_full[par], n_unit >> 1 & 1)) break;
        // ---- the CTA's sums to every CTA of the cluster, then the row log-sum-exp ----
        {
          float mw[2], tw[2];                       // 16 / n_cb warps share a column: two for each of its threads
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int x = sub + i * tpc, ew = 4 * (col / kNC + n_cb * (x >> 2)) + (x & 3);
            mw[i] = aux->warp_part[par][ew][col & (kNC - 1)][0];
            tw[i] = aux->warp_part[par][ew][col & (kNC - 1)][1];
          }
          float m = fmaxf(mw[0], mw[1]);
#pragma unroll
          for (int d = 1; d < tpc; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
          float t = (tw[0] == 0.f ? 0.f : tw[0] * ex2(mw[0] - m)) + (tw[1] == 0.f ? 0.f : tw[1] * ex2(mw[1] - m));
#pragma unroll
          for (int d = 1; d < tpc; d <<= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
          const float l = t == 0.f ? kNegInf : m + log2f(t);
          if (n_cta == 1) {                         // alone (a launch without clusters has no st.async)
            if (sub == 0) aux->part[par][0][col] = l;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&aux->sum_bar));
            wait_for(aux->sum_bar, n_unit & 1);
          } else {
            for (int p = sub; p < (int)n_cta; p += tpc)
              peer_store_async(peer_addr(smem_u32(&aux->part[par][rank][col]), p), l, peer_addr(smem_u32(&aux->part_full[par]), p));
            ok = cluster_wait(smem_u32(&aux->part_full[par]), n_unit >> 1 & 1, abort_flag, kPolls) && ok;
            ok = __all_sync(0xFFFFFFFFu, ok);
          }
          if (!ok) break;
        }
        // every warp by itself, which spares the group a barrier
        bool by_value = aux->any_kept[par] == n_unit + 1;
#pragma unroll
        for (int c0 = 0; c0 < NP; c0 += 32) {
          const int c = c0 + lane;
          if (NP < 32 && c >= NP) break;
          float l[kMaxCluster], m = kNegInf, t = 0.f;
#pragma unroll
          for (int p = 0; p < kMaxCluster; ++p) {
            l[p] = p < (int)n_cta ? aux->part[par][p][c] : kNegInf;
            m = fmaxf(m, l[p]);
          }
#pragma unroll
          for (int p = 0; p < kMaxCluster; ++p) t += ex2(l[p] - m);                       // -inf: adds nothing
          const float lse2 = m + log2f(t);
          aux->nlse[st >> 5][c] = c < w.nv ? -lse2 : kNegInf;
          const bool tiny = lse2 > 126.f;
          const float f = ex2(lse2 < -126.f ? 126.f : tiny ? -0.5f * lse2 : -lse2);       // beyond 2^126 no column is below 2^100
          aux->factor[st >> 5][c] = c < w.nv ? f : 0.f;
          aux->factor2[st >> 5][c] = tiny ? f : 1.f;
          by_value = by_value || (c < w.nv && !(lse2 <= 126.f));
          if (rank == 0 && st < 32 && c < w.nv && a.lse_nat_out)
            a.lse_nat_out[((size_t)w.layer * s.Hq + w.h) * s.T + w.t0 + w.q0 + c] = lse2 * 0.69314718055994530942f;
        }
        by_value = __any_sync(0xFFFFFFFFu, by_value);
        __syncwarp();
        // armed again for the unit after the next: a peer sends that only when it has this CTA's sums of the next unit
        if (st == 0 && n_cta > 1) mbar_expect_tx(smem_u32(&aux->part_full[par]), n_cta * NP * 4);

        const bool last = unit_from(u + unit_step) >= a.n_units;      // then step 1's groups take four tiles of five
        if (last) {
          if (st == 0) aux->last_by_value = by_value;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&aux->last_unit));
        }
        const int j_all = last ? 5 : 1;             // this group's tiles: every j_all-th
        tc_fence_after();
        auto finish = [&](int j, float total) {     // the tile's accumulator goes back, its sums go out
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&aux->acc_empty[slot_of(j)]));
          store(w, j, total);
        };
        if (!by_value) {
          // pieces of 16 columns, the load of the next one in flight while one is added
          const float4* f4 = reinterpret_cast<const float4*>(aux->factor[st >> 5]);
          uint32_t x[2][kNC];
          if (w.n > 0) {
            tmem_ld16(t_lane + slot_of(0) * NP, x[0]);
            tmem_wait16(x[0]);
          }
          for (int j = 0; j < w.n; j += j_all) {
            const bool more = j + j_all < w.n;
            f32x2 acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
            for (int b = 0; b < n_cb; ++b) {
              if (b + 1 < n_cb) tmem_ld16(t_lane + slot_of(j) * NP + (b + 1) * kNC, x[(b + 1) & 1]);
              else if (more) tmem_ld16(t_lane + slot_of(j + j_all) * NP, x[(b + 1) & 1]);
#pragma unroll
              for (int i = 0; i < kNC / 4; ++i) {
                const float4 f = f4[b * (kNC / 4) + i];
                acc[2 * (i & 1)] = fma2(pack2(x[b & 1][4 * i], x[b & 1][4 * i + 1]), pack2f(f.x, f.y), acc[2 * (i & 1)]);
                acc[2 * (i & 1) + 1] = fma2(pack2(x[b & 1][4 * i + 2], x[b & 1][4 * i + 3]), pack2f(f.z, f.w), acc[2 * (i & 1) + 1]);
              }
              if (b + 1 < n_cb) tmem_wait16(x[(b + 1) & 1]);
            }
            const f32x2 sums[2] = {add2(acc[0], acc[2]), add2(acc[1], acc[3])};
            finish(j, sum4(sums));
            if (more) {
              tmem_wait16(x[n_cb & 1]);
              if constexpr (n_cb == 1) {
#pragma unroll
                for (int i = 0; i < kNC; ++i) x[0][i] = x[1][i];
              }
            }
          }
        } else {
          for (int j = 0; j < w.n; j += j_all) finish(j, by_value_tile(w, j, par, st >> 5));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&aux->sums_empty[par]));
        n_acc += w.n;
        ++n_unit;
      }
      if (st == 0) aux->n_unit = n_unit;
    }
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
template <int D, int NP, uint32_t kPolls>
int resident_clusters(int log_cta, int smem) {
  static std::atomic<int> known[kMaxDevices][4];
  auto kern = score_window_kernel<D, NP, kPolls>;
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

template <int D, int NP, uint32_t kPolls>
int launch_window_polls(const CUtensorMap& mq, const CUtensorMap& mk, const WinArgs& a, int units, int log_cta, cudaStream_t stream) {
  constexpr int smem = kSmemTiles * kTile * D * 2 + kAuxBytes + 1024;
  auto kern = score_window_kernel<D, NP, kPolls>;
  const int clusters = resident_clusters<D, NP, kPolls>(log_cta, smem);
  if (clusters < 1) return KVCRUSH_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return KVCRUSH_ERR_CUDA;
  const int n = clusters < units ? clusters : units;
  return launch_chained(kern, dim3((unsigned)n << log_cta), dim3(kThreads), smem, stream, 1 << log_cta, mq, mk, a);
}

template <int D, int NP>
int launch_window(const CUtensorMap& mq, const CUtensorMap& mk, const WinArgs& a, int units, int log_cta, bool short_waits,
                  cudaStream_t stream) {
  return short_waits ? launch_window_polls<D, NP, kShortWaitPolls>(mq, mk, a, units, log_cta, stream)
                     : launch_window_polls<D, NP, kWaitPolls>(mq, mk, a, units, log_cta, stream);
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
  const int n_pad = pad_window(s.window);
  a.ring = kMaxRing;                                // two query buffers of n_pad rows take the sixth tile at most
  CUtensorMap mq;
  if (!make_map(&mq, Q, s.D, s.T, s.Hq, s.n_layers, n_pad)) return KVCRUSH_ERR_UNSUPPORTED;
  const CUtensorMap& mk = *reinterpret_cast<const CUtensorMap*>(maps.k);
  const bool sw = diag.short_waits != 0;
  auto launch = s.D > 64 ? (n_pad == 16 ? launch_window<128, 16> : n_pad == 32 ? launch_window<128, 32> : launch_window<128, 64>)
                         : (n_pad == 16 ? launch_window<64, 16> : n_pad == 32 ? launch_window<64, 32> : launch_window<64, 64>);
  const int n_sms = sm_count();
  const Plan plan = plan_launches(s, cu_host, n_sms, n_pad);
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

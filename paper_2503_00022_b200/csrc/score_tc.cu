// Stage 1 on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), bf16 or fp16 Q/K, head_dim up to 128
// (a multiple of 8; widths other than 64 and 128 run in the next larger kernel: the TMA boxes read zeros past
// the last channel, and zeros add nothing to a dot product).
//
// Attention column sums (Algorithm 1 of the paper: A_h = softmax(Q_h K_h^T / sqrt(d_k)), then the per-token
// sum of A_h over the queries) without ever storing the S x S matrix: two sweeps that both recompute
// 128 x 128 logit tiles.
//
//   sweep 1 (kColsum = false)  S = Q_block K^T: TMEM lane = query row, so each epilogue thread owns one row
//                              and keeps its running (max, sum) in registers -> lse2(j) = log2 sum_t 2^(s2(j,t))
//   sweep 2 (kColsum = true)   S^T = K_block Q^T: TMEM lane = key, so each epilogue thread owns one key column
//                              and adds 2^(s2 - lse2(j)) = A(j, t) over all query tiles in registers.
//                              No shuffles or atomics: one deterministic store per key.
//   s2 = q.k * softmax_scale * log2(e).
//
// On this part the sweeps run against the board's power limit, so the work decomposition is built to
// spend little energy per logit tile:
//
//   * one CTA per SM lives for the whole launch and pulls work items from an atomic counter, so TMEM
//     allocation, barrier set-up and pipeline fill are paid once per SM instead of once per item;
//   * an item is a 512-row block of the stationary operand (four 128-row quarters; fewer when a launch has few
//     items, see block_tiles).  Every streamed 128-row tile is multiplied with all four quarters, which quarters
//     the L2 -> shared-memory traffic per logit compared with one tile pair per load;
//   * TMEM holds one 128-column accumulator per quarter, owned by one epilogue group: a group needs no merge
//     with another group, and while it waits for its accumulator to be refilled the other three keep the
//     special-function unit busy.
//
// Roles: warp 0 fetches + decodes items and issues TMA loads; warps 1 and 2 (one lane each) issue the
// tcgen05.mma of quarters 0-1 and 2-3; warp 3 overwrites the queries of the column sweep's streamed tiles that do not
// vote (see there) and idles in the row sweep; warps 4..19 are four epilogue groups (one per quarter) of 128 threads,
// thread = TMEM lane = one query row (sweep 1) or one key column (sweep 2).  All synchronisation is by mbarriers
// with bounded waits: a role that gives up sets the CTA's abort flag, every other wait then ends, the CTA
// reports through the status word, drains its copies, frees TMEM and returns.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace kvc {

namespace {

using namespace tc;

constexpr int kTile = 128;
constexpr int kQ = 4;                        // stationary 128-row quarters per work item
constexpr int kEpiWarps = 16;
#ifndef KVC_ISSUE_WARPS
#define KVC_ISSUE_WARPS 2
#endif
constexpr int kIssueWarps = KVC_ISSUE_WARPS;   // tcgen05.mma issuing threads; each owns kQ / kIssueWarps quarters
constexpr int kQPerIssuer = kQ / kIssueWarps;
constexpr int kCtrlWarps = 4;                // one warpgroup: producer, issuers, the warp for non-voting queries
constexpr int kEdgeWarp = 3;
constexpr int kThreads = 32 * (kCtrlWarps + kEpiWarps);
// Registers: 96 a thread at launch (the most 20 warps can have); the control warpgroup gives some back (what its roles
// need in either sweep) and the epilogue takes 104.
template <bool kColsum> constexpr int kCtrlRegs = kColsum ? 64 : 48;
constexpr int kEpiRegs = 104;
static_assert(kIssueWarps < kEdgeWarp && 32 * kCtrlWarps * kCtrlRegs<true> + 32 * kEpiWarps * kEpiRegs <= kThreads * 96,
              "register split within the launch's total");
constexpr int kTiles = 6;                    // 128-row tiles in shared memory: tpb stationary ones, the others a ring of streamed tiles
constexpr int kMaxRing = kTiles - 1;
constexpr uint32_t kTmemCols = 512;          // one 128-column fp32 accumulator per quarter
constexpr int kLseChunk = 16;                // sweep 2: streamed tiles whose row log-sum-exp is staged at once
// Items announced ahead.  The epilogue holds an item until its results are written; where items are single tiles (the row
// sweep of sequences of one tile, the one use of that instantiation) two are too few to hide the next one's fetch.  In the
// other sweeps four cost 1 to 2 % (8 layers x 32 heads x 8192 tokens 4.70 against 4.78 ms).
constexpr int kMaxItemSlots = 4;
template <bool kColsum, bool kSplit> constexpr int kItemSlots = kColsum || kSplit ? 2 : kMaxItemSlots;

struct PersistArgs {
  Shape s;
  float scale_log2;
  const float* lse;        // sweep 2: row log-sum-exp; value * lse_mul is in the log2 domain
  float lse_mul;
  float* lse2_out;         // sweep 1 output (log2 domain), [n_layers][Hq][T]
  float* lse_nat_out;      // sweep 1: optional natural-log copy
  float* scores;           // sweep 2 output
  int normalize;
  int bf16;                // operand type of Q and K: bf16 (1) or fp16 (0)
  int tpb;                 // 128-row tiles of an item's stationary block: 4, or 2 or 1 when the launch has few items
  int max_blocks;          // ceil(max_seqlen / (tpb * kTile))
  int n_items;             // (sequence, stationary block) pairs of one (layer, head)
  int total_items;         // n_items * n_layers * Hq
  int n_lh;                // n_layers * Hq
  int tail_lh;             // the last tail_lh (layer, head) pairs are handed out heaviest item first across all of them
  int* counter;            // work counter, zero at launch; NULL: items are dealt out in advance (see the producer)
  int32_t* status;
  int withhold_first_item; // diagnostic: the producer warp fetches its first item and then stops before announcing
                           // it or issuing any copy for it, so that every consumer's first wait runs out (2: in the first
                           // CTA of the row sweep only)
};

template <int D>
struct PSmem {
  static constexpr int kTileBytes = kTile * D * 2;
  static constexpr int kBlockBytes = kTile * 128;
  static constexpr int kAuxOff = kTiles * kTileBytes;           // the stationary quarters, then the ring, from offset 0
  static constexpr int kAuxBytes = 26624;
  static constexpr int kTotal = kAuxOff + kAuxBytes + 1024;
};

struct PAux {
  unsigned long long full[kMaxRing], empty[kMaxRing];
  unsigned long long edge_full[kMaxRing];             // sweep 2: a tile with queries that do not vote has landed
  unsigned long long fixed_full, fixed_empty;
  unsigned long long acc_full[kQ], acc_empty[kQ];     // [quarter]
  unsigned long long item_full[kMaxItemSlots], item_empty[kMaxItemSlots];
  unsigned long long epi_bar;                         // all epilogue warps (sweep 2: a chunk of -lse2 is in place;
                                                      // sweep 1 with an observation window: slots merge)
  unsigned long long drain[kIssueWarps];
  uint32_t tmem_base;
  int abort_flag;
  int item[kMaxItemSlots][8];                                     // layer, head, first tile, tiles, first token, tokens (layer < 0: no more work)
  alignas(16) float lse_chunk[2][kLseChunk * kTile];  // [buffer][streamed tile inside the chunk][query]: minus lse2
  alignas(16) float part[2][kQ][2][kTile];            // [item parity][slot][max, sum][row]: sweep 1, replicated quarters
};

// Geometry of one work item, derived identically by every role.
template <bool kColsum, bool kSplit>
struct Geo {
  int layer, h, hk, t0, L, first_stream, n_iter;
  int row0, tile0;             // first row of the stationary block inside the sequence, and row0 / kTile
  int ws;                      // first query row that votes (0 without an observation window)
  bool last_seq;               // nothing is packed behind the sequence: TMA reads zeros past its end
  bool causal;
  int nq;                      // 128-row quarters of the block that hold rows of the sequence
  // The four accumulator slots normally hold four quarters.  When an item has only one or two (small blocks, the last
  // block of a sequence, in sweep 1 also an observation window whose queries lie in one or two quarters), each quarter
  // serves rep = 4 or 2 slots and slot s takes the streamed tiles it with it % rep == s % rep, so that all four epilogue
  // groups stay busy; the slots' sums are merged at the end of the item.  (kSplit; without it rep is the constant 1.)
  int rep, v0;                 // slots per quarter; first quarter with work
  __device__ __forceinline__ Geo(const Shape& s, const volatile int* it, int tpb) {
    layer = it[0]; h = it[1]; tile0 = it[2]; t0 = it[4]; L = it[5];
    const int n_tiles = it[3];
    hk = h / s.G;
    row0 = tile0 * kTile;
    causal = s.causal != 0;
    nq = min(tpb, (L - row0 + kTile - 1) / kTile);
    ws = (s.window > 0 && L > s.window) ? L - s.window : 0;
    last_seq = t0 + L == s.T;
    v0 = 0;
    if (kColsum) {                                                      // stationary keys, streamed query tiles
      first_stream = max(causal ? tile0 : 0, ws / kTile);
      n_iter = n_tiles - first_stream;
    } else {                                                            // stationary queries, streamed key tiles
      first_stream = 0;
      n_iter = causal ? min(tile0 + tpb, n_tiles) : n_tiles;
      if (ws > row0) v0 = min(nq - 1, (ws - row0) / kTile);
    }
    rep = !kSplit ? 1 : nq - v0 == 1 ? 4 : nq - v0 == 2 ? 2 : 1;
  }
  // Sweep 2: the rows [lo, end) of streamed tile i hold queries that vote (or zeros); the others belong to the next sequence or
  // come before the window.  Only the first and the last tile of an item can have such rows.
  struct Voters { int lo, end; __device__ __forceinline__ bool all() const { return lo == 0 && end == kTile; } };
  __device__ __forceinline__ Voters voters(int i) const {
    const int j0 = (first_stream + i) * kTile;
    return {max(0, ws - j0), last_seq ? kTile : min(kTile, L - j0)};
  }
  __device__ __forceinline__ int quarter(int slot) const { return rep > 1 ? v0 + slot / rep : slot; }
  // Streamed tiles of a slot: first, first + rep, .. below end; `diag`: the one that holds the causal diagonal (-1: none).
  struct Range { int first, end, diag; };
  __device__ __forceinline__ Range range(int slot) const {
    const int qd = quarter(slot), rr = slot & (rep - 1), own = tile0 + qd - first_stream;
    if (qd >= nq || qd < v0) return {0, 0, -1};                         // no rows, or no voting query
    if (!causal) return {rr, n_iter, -1};
    if (!kColsum) return {rr, min(n_iter, own + 1), own};
    const int lo = max(own, 0);
    return {lo + ((rr - lo) & (rep - 1)), n_iter, own};
  }
};

// kSplit: items with one or two quarters spread them over all four accumulators.  The column sweep has an instantiation
// without it for full blocks: carrying it along costs 2 % there (372 against 365 us at 2 layers of 5003 + 3117 tokens,
// 4 % at ragged 500 to 1000 tokens), while its partial last blocks are its lightest items.
// D: channels of a tile in shared memory (64 or 128); kSteps: 16-channel steps of a dot product that are multiplied (heads
// of 65 to 96 channels: 6 of 8, the rest is zeros: heads of 96, one sweep of 5003 + 3117 tokens x 8 layers 1418 -> 1355 us;
// as a run-time bound it cost the full width 0.5 %).
// kEarly: a column sweep right behind its row sweep.  Only its epilogue waits for the row log-sum-exp; items, loads and the
// first products read the call's inputs and start as soon as an SM is free.
// kEdge: a column sweep some of whose tiles hold queries that do not vote (see the edge warp).
// kPolls: polls of every bounded barrier wait (a compile-time constant: the epilogue has no register to spare for it).
template <int D, int kSteps, bool kColsum, bool kSplit, bool kEarly, bool kEdge, uint32_t kPolls>
__global__ void __launch_bounds__(kThreads, 1)
score_persist_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const PersistArgs a) {
  using SL = PSmem<D>;
  constexpr int kSlots = kItemSlots<kColsum, kSplit>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  PAux* aux = reinterpret_cast<PAux*>(smem + SL::kAuxOff);
  volatile int* abort_flag = &aux->abort_flag;
  const int ring = kTiles - a.tpb;
  const uint32_t fixed_addr = smem_u32(smem), ring_addr = fixed_addr + a.tpb * SL::kTileBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Shape& s = a.s;

  if (warp == 0) {
    if (lane == 0) {
      for (int i = 0; i < kMaxRing; ++i) { mbar_init(smem_u32(&aux->full[i]), 1); mbar_init(smem_u32(&aux->empty[i]), kIssueWarps); mbar_init(smem_u32(&aux->edge_full[i]), 1); }
      mbar_init(smem_u32(&aux->fixed_full), 1);
      mbar_init(smem_u32(&aux->fixed_empty), kIssueWarps);
      for (int i = 0; i < kIssueWarps; ++i) mbar_init(smem_u32(&aux->drain[i]), 1);
      for (int i = 0; i < kQ; ++i) {
        mbar_init(smem_u32(&aux->acc_full[i]), 1);
        mbar_init(smem_u32(&aux->acc_empty[i]), 4);
      }
      mbar_init(smem_u32(&aux->epi_bar), kEpiWarps);
      for (int i = 0; i < kSlots; ++i) {
        mbar_init(smem_u32(&aux->item_full[i]), 1);
        mbar_init(smem_u32(&aux->item_empty[i]), kIssueWarps + kEpiWarps + (kEdge ? 1 : 0));
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  } else if (warp == 1) {
    tmem_alloc(smem_u32(&aux->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  if constexpr (!kEarly) {
    chain_wait();
    chain_trigger();
  }
  // a launch that already failed somewhere is not worth finishing
  if (tid == 0) aux->abort_flag = *reinterpret_cast<volatile int32_t*>(a.status) != 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = aux->tmem_base;
  const bool dead = aux->abort_flag != 0;

  const CUtensorMap* map_fixed = kColsum ? &map_k : &map_q;
  const CUtensorMap* map_stream = kColsum ? &map_q : &map_k;

  if (dead) {
    if constexpr (kEarly) chain_wait();            // the row sweep's other CTAs may still run: no later kernel may start beside them
  } else if (warp < kCtrlWarps) {
  set_max_regs<kCtrlRegs<kColsum>, false>();
  if (warp == 0) {
    // ------------------------------ work fetch + TMA producer ------------------------------
    int n_item = 0, n_stream = 0;     // n_stream: streamed tiles issued
    int rs = 0;                       // lane 0: ring slot of the next tile
    uint32_t ring_phase = 0;          //         and its phase
    uint32_t edge_last = 0, edge_phase = 0;   // lane 0, bit per ring slot: its tile is announced by edge_full; phase of that
    int issued_item = 0;              // lane 0: items whose stationary load was issued
    bool alive = true;
    while (alive) {
      const int slot = n_item % kSlots;
      int idx = 0;
      bool ok = true;
      if (lane == 0) {
        ok = mbar_wait(smem_u32(&aux->item_empty[slot]), ((n_item / kSlots) & 1) ^ 1, abort_flag, kPolls);
        // Up to two items a block: dealt out in advance, heaviest first in snake order (block b takes b and 2n - 1 - b), which
        // spares the call the memset of the counter.
        if (ok) idx = a.counter ? atomicAdd(a.counter, 1)
                                : n_item * (int)gridDim.x + (n_item & 1 ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x);
      }
      ok = __shfl_sync(0xFFFFFFFFu, (int)ok, 0) != 0;
      idx = __shfl_sync(0xFFFFFFFFu, idx, 0);
      if (!ok) break;
      if (idx >= a.total_items) {
        if (lane == 0) { aux->item[slot][0] = -1; mbar_arrive(smem_u32(&aux->item_full[slot])); }
        break;
      }
      if (a.withhold_first_item == 1 || (a.withhold_first_item && !kColsum && blockIdx.x == 0)) break;   // nothing is in flight: the consumers' bounded waits end the CTA
      // (layer, head)-major order keeps the CTAs that run together on a few heads (their Q and K stay in L2); the
      // last pairs are taken weight-major instead, so that the launch does not end with a few CTAs on the heaviest
      // items of the last head while the others idle (a launch with few items is all tail)
      int lh, rank;
      const int head_part = (a.n_lh - a.tail_lh) * a.n_items;
      if (idx < head_part) {
        lh = idx / a.n_items; rank = idx - lh * a.n_items;
      } else {
        const int j = idx - head_part;
        rank = j / a.tail_lh; lh = a.n_lh - a.tail_lh + (j - rank * a.tail_lh);
      }
      int seq, blk, nblk;
      decode_item(s.cu_seqlens, s.n_seqs, a.max_blocks, rank, !kColsum, lane, seq, blk, nblk, a.tpb * kTile, s.window);
      if (lane == 0) {
        int* it = aux->item[slot];
        it[0] = lh / s.Hq; it[1] = lh - it[0] * s.Hq; it[2] = blk * a.tpb;
        it[4] = __ldg(s.cu_seqlens + seq); it[5] = __ldg(s.cu_seqlens + seq + 1) - it[4];
        it[3] = (it[5] + kTile - 1) / kTile;
        mbar_arrive(smem_u32(&aux->item_full[slot]));
        const Geo<kColsum, kSplit> g(s, it, a.tpb);
        const int head_fixed = kColsum ? g.hk : g.h, head_stream = kColsum ? g.h : g.hk;
        // the stationary buffer is free once every MMA of the previous item has retired
        ok = mbar_wait(smem_u32(&aux->fixed_empty), (n_item & 1) ^ 1, abort_flag, kPolls);
        if (ok) {
          const int n_fixed = g.nq - g.v0;
          mbar_expect_tx(smem_u32(&aux->fixed_full), n_fixed * SL::kTileBytes);
          for (int q = 0; q < n_fixed; ++q)
#pragma unroll
            for (int kb = 0; kb < D / 64; ++kb)
              tma_load_4d(fixed_addr + q * SL::kTileBytes + kb * SL::kBlockBytes, map_fixed, smem_u32(&aux->fixed_full),
                          kb * 64, g.t0 + g.row0 + (g.v0 + q) * kTile, head_fixed, g.layer);
          issued_item = n_item + 1;
          for (int i = 0; ok && i < g.n_iter; ++i) {
            ok = mbar_wait(smem_u32(&aux->empty[rs]), ring_phase ^ 1, abort_flag, kPolls);
            if (!ok) break;
            uint32_t landed = smem_u32(&aux->full[rs]);
            if constexpr (kEdge) {                 // edge_full first, the edge warp passes it on to `full`
              edge_last &= ~(1u << rs);
              if (!g.voters(i).all()) {
                landed = smem_u32(&aux->edge_full[rs]);
                edge_last |= 1u << rs;
                edge_phase ^= 1u << rs;
              }
            }
            mbar_expect_tx(landed, SL::kTileBytes);
#pragma unroll
            for (int kb = 0; kb < D / 64; ++kb)
              tma_load_4d(ring_addr + rs * SL::kTileBytes + kb * SL::kBlockBytes, map_stream, landed,
                          kb * 64, g.t0 + (g.first_stream + i) * kTile, head_stream, g.layer);
            ++n_stream;
            if (++rs == ring) { rs = 0; ring_phase ^= 1; }
          }
        }
      }
      alive = __shfl_sync(0xFFFFFFFFu, (int)ok, 0) != 0;
      n_stream = __shfl_sync(0xFFFFFFFFu, n_stream, 0);
      ++n_item;
    }
    if (lane == 0 && *abort_flag) {
      // give the copies in flight a bounded time to land before the CTA's shared memory is released
      for (int q = max(0, n_stream - ring); q < n_stream; ++q) {
        const int slot = q % ring;
        const bool edge = kEdge && (edge_last >> slot & 1u);
        const uint32_t bar = smem_u32(edge ? &aux->edge_full[slot] : &aux->full[slot]);
        const uint32_t parity = edge ? (edge_phase >> slot & 1u) ^ 1u : (uint32_t)(q / ring) & 1u;
        for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(bar, parity); ++i) {}
      }
      if (issued_item > 0)
        for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(smem_u32(&aux->fixed_full), (issued_item - 1) & 1); ++i) {}
    }
  } else if (warp <= kIssueWarps) {
    // ------------------------------ MMA issuers ------------------------------
    // One thread per pair of stationary quarters.  tcgen05.mma blocks its issuer while the tensor core's queue is
    // full, and the queue is short, so a lone issuer leaves the pipe idle whenever it has to poll a barrier; with
    // two issuers one polls while the other's instructions are queued.
    if (lane == 0) {
      const int iw = warp - 1;
      const uint32_t idesc = make_idesc(kTile, kTile, a.bf16 != 0);
      int n_item = 0, rs = 0, cnt[kQPerIssuer] = {};
      uint32_t ring_phase = 0;
      bool ok = true;
      while (ok) {
        const int slot = n_item % kSlots;
        ok = mbar_wait(smem_u32(&aux->item_full[slot]), (n_item / kSlots) & 1, abort_flag, kPolls);
        if (!ok) break;
        const volatile int* it = aux->item[slot];
        if (it[0] < 0) break;
        const Geo<kColsum, kSplit> g(s, it, a.tpb);
        mbar_arrive(smem_u32(&aux->item_empty[slot]));
        ok = mbar_wait(smem_u32(&aux->fixed_full), n_item & 1, abort_flag, kPolls);
        typename Geo<kColsum, kSplit>::Range rg[kQPerIssuer];
        uint32_t a_addr[kQPerIssuer];
#pragma unroll
        for (int u = 0; u < kQPerIssuer; ++u) {
          rg[u] = g.range(kQPerIssuer * iw + u);
          a_addr[u] = fixed_addr + (g.quarter(kQPerIssuer * iw + u) - g.v0) * SL::kTileBytes;
        }
        for (int i = 0; ok && i < g.n_iter; ++i) {
          // also when its quarters skip the tile: the wait keeps the issuer from running a whole ring ahead of
          // the other one, whose arrival on empty[rs] must fall into the same phase as this one's
          ok = mbar_wait(smem_u32(&aux->full[rs]), ring_phase, abort_flag, kPolls);
          if (!ok) break;
#pragma unroll
          for (int u = 0; u < kQPerIssuer; ++u) {
            if (!ok) break;
            const int qd = kQPerIssuer * iw + u;
            if (i < rg[u].first || i >= rg[u].end || ((i - rg[u].first) & (g.rep - 1))) continue;
            const int c = cnt[u]++;                 // the quarter's accumulator is reused every time: phase c & 1
            ok = mbar_wait(smem_u32(&aux->acc_empty[qd]), (c & 1) ^ 1, abort_flag, kPolls);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + qd * kTile;
#pragma unroll
            for (int k = 0; k < kSteps; ++k) {
              const uint32_t off = (k >> 2) * SL::kBlockBytes + (k & 3) * 32;
              umma_bf16(d_tmem, smem_desc_sw128(a_addr[u] + off),
                        smem_desc_sw128(ring_addr + rs * SL::kTileBytes + off), idesc, k > 0);
            }
            umma_commit(smem_u32(&aux->acc_full[qd]));
          }
          if (!ok) break;
          // this issuer is done with the ring slot (a commit with nothing pending arrives at once)
          umma_commit(smem_u32(&aux->empty[rs]));
          if (++rs == ring) { rs = 0; ring_phase ^= 1; }
        }
        if (!ok) break;
        umma_commit(smem_u32(&aux->fixed_empty));
        ++n_item;
      }
      if (*abort_flag) {
        // wait (bounded) until every MMA already issued has retired before TMEM and shared memory go away
        umma_commit(smem_u32(&aux->drain[iw]));
        for (uint32_t i = 0; i < kDrainPolls && !mbar_try_wait(smem_u32(&aux->drain[iw]), 0); ++i) {}
      }
    }
  } else if (kEdge && warp == kEdgeWarp) {
    // ------------------------------ queries that do not vote ------------------------------
    // A weight of 2^(x - inf) is 0 only while x is finite or -inf: a NaN or an infinite logit of the next sequence's first
    // queries, or of one before the window, would reach every key of the block.  So their rows take the values of the tile's
    // last query that votes before the products are formed: it sees every key whose sum this tile adds to, so that what is
    // not finite then is not finite in its own right.  (Masked in the epilogue instead, which has no instruction to spare:
    // heads of 96, 5003 + 3117 tokens, both sweeps 2546 -> 2634 us, 64 sequences of 130 tokens 3884 -> 4380, and 1 % where there
    // is nothing to mask.)  The detour from the tile's landing over this warp to the issuers takes about half a us, which is
    // seen where an item has one or two tiles: 22 layers x 32 heads, 383 tokens, window of 128, 71.9 -> 76.1 us, 27 layers of
    // 269 + 110 tokens with a given log-sum-exp, whole pass, 82.3 -> 86.9; batches of 500 to 4000 tokens 0 to 1 %.  (The first
    // tile loaded before the stationary ones hides it for windows, 74.1 us, and costs the others 1 %.)
    int n_item = 0, rs = 0;
    uint32_t phase = 0;               // bit per ring slot: phase of edge_full
    bool ok = true;
    while (ok) {
      const int slot = n_item % kSlots;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&aux->item_full[slot]), (n_item / kSlots) & 1, abort_flag, kPolls));
      if (!ok) break;
      const volatile int* it = aux->item[slot];
      if (it[0] < 0) break;
      const Geo<kColsum, kSplit> g(s, it, a.tpb);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&aux->item_empty[slot]));
      for (int i = 0; i < g.n_iter; i += max(1, g.n_iter - 1)) {         // the first and the last tile
        const auto v = g.voters(i);
        if (v.all()) continue;
        const int q = (rs + i) % ring;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&aux->edge_full[q]), phase >> q & 1u, abort_flag, kPolls));
        if (!ok) break;
        phase ^= 1u << q;
        // a lane keeps one 16-byte piece of every 64 channels; the swizzle has piece c of row r at place c ^ (r & 7)
        const uint32_t tile = ring_addr + q * SL::kTileBytes;
        const int piece = lane & 7, from = v.end - 1;
        uint4 val[D / 64];
#pragma unroll
        for (int kb = 0; kb < D / 64; ++kb) val[kb] = ld_shared16(tile + kb * SL::kBlockBytes + from * 128 + ((piece ^ (from & 7)) << 4));
        auto fill = [&](int first, int end) {
#pragma unroll 8
          for (int row = first + (lane >> 3); row < end; row += 4)
#pragma unroll
            for (int kb = 0; kb < D / 64; ++kb) st_shared16(tile + kb * SL::kBlockBytes + row * 128 + ((piece ^ (row & 7)) << 4), val[kb]);
        };
        fill(0, v.lo);
        fill(v.end, kTile);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // read by tcgen05.mma
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&aux->full[q]));
      }
      rs = (rs + g.n_iter) % ring;
      ++n_item;
    }
  }
  } else {
    // ------------------------------ epilogue groups ------------------------------
    set_max_regs<kEpiRegs, true>();
    const int gi = (warp - kCtrlWarps) >> 2;  // group = stationary quarter; it owns that quarter's accumulator
    const int quarter = warp & 3;                  // TMEM lanes this warp may read
    const int r = quarter * 32 + lane;             // row of the accumulator = TMEM lane = index inside the group
    const uint32_t t_acc = tmem_base + ((uint32_t)(quarter * 32) << 16) + gi * kTile;
    const uint32_t acc_full = smem_u32(&aux->acc_full[gi]), acc_empty = smem_u32(&aux->acc_empty[gi]);
    const float scale = a.scale_log2;
    const f32x2 scale2 = splat2(scale);
    const float ninf = __int_as_float(0xFF800000);
    int n_item = 0, cnt = 0, n_esync = 0, n_merge = 0;
    bool ok = true;

    // barrier among all 16 epilogue warps; bounded like every other wait
    auto epi_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&aux->epi_bar));
      ok = mbar_wait(smem_u32(&aux->epi_bar), n_esync & 1, abort_flag, kPolls) && ok;
      ++n_esync;
    };
    auto release = [&]() {                         // accumulator drained: hand it back to its issuer
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    };

    if constexpr (kEarly) {                        // the row log-sum-exp is complete, unless its sweep gave up
      chain_wait();
      chain_trigger();
      if (*reinterpret_cast<volatile int32_t*>(a.status) != 0) { *abort_flag = 1; ok = false; }
    }
    while (true) {
      const int slot = n_item % kSlots;
      ok = mbar_wait(smem_u32(&aux->item_full[slot]), (n_item / kSlots) & 1, abort_flag, kPolls) && ok;
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) break;
      // The item is read again when its results are written, rather than kept in registers, of which there is none to
      // spare; the slot is handed back after that.
      const volatile int* it = aux->item[slot];
      if (it[0] < 0) break;
      const Geo<kColsum, kSplit> g(s, it, a.tpb);
      const auto rg = g.range(gi);

      if constexpr (kColsum) {
        const float* lse_row = a.lse + ((size_t)g.layer * s.Hq + g.h) * s.T + g.t0;
        // Minus lse2 of the streamed queries reaches the epilogue threads through shared memory, kLseChunk tiles
        // at a time and once for all four groups: all 16 warps fill the next chunk's buffer, then work through the
        // current chunk, and meet once per chunk (the buffer of chunk k is rewritten as chunk k + 2 only after
        // everybody left chunk k).
        const int et = tid - 32 * kCtrlWarps;
        auto fill = [&](int k) {
          float* dst = aux->lse_chunk[k & 1];
#pragma unroll
          for (int e = et; e < kLseChunk * kTile; e += kEpiWarps * 32) {
            const int i = kLseChunk * k + (e >> 7);
            const int j = (g.first_stream + i) * kTile + (e & (kTile - 1));
            dst[e] = (i < g.n_iter && j < g.L && j >= g.ws) ? -((kEarly ? __ldcg(lse_row + j) : __ldg(lse_row + j)) * a.lse_mul) : ninf;
          }
        };
        f32x2 acc[2] = {0ull, 0ull};
        const int n_chunks = (g.n_iter + kLseChunk - 1) / kLseChunk;
        int i = rg.first;
        fill(0);
        epi_sync();
        for (int k = 0; k < n_chunks && ok; ++k) {
          if (k + 1 < n_chunks) fill(k + 1);
          const int i_end = min(rg.end, kLseChunk * (k + 1));
          for (; i < i_end; i += g.rep) {
            const int c = cnt++;
            const float* lse_buf = aux->lse_chunk[k & 1] + (i & (kLseChunk - 1)) * kTile;
            ok = mbar_wait(acc_full, c & 1, abort_flag, kPolls) && ok;
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            tc_fence_after();
            if (i == rg.diag)
              sweep_tile<true>(t_acc, [&](const uint32_t (&v)[16], int p) { colsum_piece<true>(v, lse_buf + p * 16, scale2, r, p * 16, acc); }, release);
            else
              sweep_tile(t_acc, [&](const uint32_t (&v)[16], int p) { colsum_piece<false>(v, lse_buf + p * 16, scale2, r, p * 16, acc); }, release);
          }
          epi_sync();
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        float total = sum4(acc);
        const Geo<kColsum, kSplit> g(s, it, a.tpb);
        const int row = g.row0 + g.quarter(gi) * kTile + r;    // token of this thread inside the sequence
        if (g.rep > 1) {                     // slots that share a quarter add up their sums
          float (*part)[2][kTile] = aux->part[n_merge++ & 1];
          part[gi][0][r] = total;
          epi_sync();
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          if ((gi & (g.rep - 1)) == 0)
            for (int u = 1; u < g.rep; ++u) total += part[gi + u][0][r];
        }
        if (row < g.L && (gi & (g.rep - 1)) == 0) {
          if (a.normalize) total = total / (float)(g.L - g.ws);
          a.scores[((size_t)g.layer * s.Hq + g.h) * s.T + g.t0 + row] = total;
        }
      } else {
        float m = __int_as_float(0xFF800000);                   // running max (log2 domain) of this row
        f32x2 sum2[2] = {0ull, 0ull};                           // packed partial sums of 2^(x - m)
        for (int i = rg.first; i < rg.end; i += g.rep) {
          const int c = cnt++;
          ok = mbar_wait(acc_full, c & 1, abort_flag, kPolls) && ok;
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          tc_fence_after();
          // keys of this tile that count for this row: up to the diagonal (causal) and inside the sequence
          const int n_valid = g.causal ? (i == rg.diag ? r + 1 : kTile) : min(kTile, g.L - i * kTile);
          // masked columns, or a row that has no reference yet (its first tile): exact maxima, piece by piece
          if (__any_sync(0xFFFFFFFFu, n_valid < kTile || !(m > -3.0e38f)))
            sweep_tile<true>(t_acc, [&](const uint32_t (&v)[16], int p) { lse_piece<true>(v, scale, scale2, n_valid - p * 16, m, sum2); }, release);
          else
            lse_tile_lazy(t_acc, scale, scale2, m, sum2, release);
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        float sum = sum4(sum2);
        const Geo<kColsum, kSplit> g(s, it, a.tpb);
        const int row = g.row0 + g.quarter(gi) * kTile + r;
        if (g.rep > 1) {                     // slots that share a quarter merge their (max, sum)
          // (alternating buffers: a slot writes one again only after the sync that follows every read of it)
          float (*part)[2][kTile] = aux->part[n_merge++ & 1];
          part[gi][0][r] = m;
          part[gi][1][r] = sum;
          epi_sync();
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          if ((gi & (g.rep - 1)) == 0) {
            float big = m;
            for (int u = 1; u < g.rep; ++u) big = fmaxf(big, part[gi + u][0][r]);
            float tot = sum == 0.f ? 0.f : sum * ex2(m - big);         // 0: a slot without tiles; NaN stays NaN
            for (int u = 1; u < g.rep; ++u) {
              const float mu = part[gi + u][0][r], su = part[gi + u][1][r];
              tot += su == 0.f ? 0.f : su * ex2(mu - big);
            }
            m = big;
            sum = tot;
          }
        }
        if (row < g.L && row >= g.ws && (gi & (g.rep - 1)) == 0) {
          const float lse2 = m + log2f(sum);
          const size_t out = ((size_t)g.layer * s.Hq + g.h) * s.T + g.t0 + row;
          a.lse2_out[out] = lse2;
          if (a.lse_nat_out) a.lse_nat_out[out] = lse2 * 0.69314718055994530942f;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&aux->item_empty[slot]));
      ++n_item;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  if (tid == 0 && !dead && *abort_flag) report(a.status, KVCRUSH_DEV_TIMEOUT, kColsum ? KID_SCORE_COLSUM : KID_SCORE_LSE, blockIdx.x, 0);
}

template <int D, int kSteps, bool kColsum, bool kSplit, bool kEarly, bool kEdge, uint32_t kPolls>
int launch_persist_polls(const CUtensorMap& mq, const CUtensorMap& mk, const PersistArgs& a, int n_sms, cudaStream_t stream) {
  auto kern = score_persist_kernel<D, kSteps, kColsum, kSplit, kEarly, kEdge, kPolls>;
  constexpr int smem = PSmem<D>::kTotal;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return KVCRUSH_ERR_CUDA;
  const int blocks = a.total_items < n_sms ? a.total_items : n_sms;
  return launch_chained(kern, dim3((unsigned)blocks), dim3(kThreads), smem, stream, 1, mq, mk, a);
}

template <bool kColsum, bool kSplit, bool kEarly, bool kEdge, uint32_t kPolls>
int launch_persist_width(const CUtensorMap& mq, const CUtensorMap& mk, const PersistArgs& a, int n_sms, cudaStream_t stream) {
  if (a.s.D <= 64) return launch_persist_polls<64, 4, kColsum, kSplit, kEarly, kEdge, kPolls>(mq, mk, a, n_sms, stream);
  if (a.s.D <= 96) return launch_persist_polls<128, 6, kColsum, kSplit, kEarly, kEdge, kPolls>(mq, mk, a, n_sms, stream);
  return launch_persist_polls<128, 8, kColsum, kSplit, kEarly, kEdge, kPolls>(mq, mk, a, n_sms, stream);
}

// edge: some tile of the column sweep holds queries that do not vote (the diagnostic build takes that kernel always)
template <bool kColsum, bool kSplit, bool kEarly = false>
int launch_persist(const CUtensorMap& mq, const CUtensorMap& mk, const PersistArgs& a, bool edge, bool short_waits, int n_sms,
                   cudaStream_t stream) {
  if (short_waits) return launch_persist_width<kColsum, kSplit, kEarly, kColsum, kShortWaitPolls>(mq, mk, a, n_sms, stream);
  return kColsum && edge ? launch_persist_width<kColsum, kSplit, kEarly, kColsum, kWaitPolls>(mq, mk, a, n_sms, stream)
                         : launch_persist_width<kColsum, kSplit, kEarly, false, kWaitPolls>(mq, mk, a, n_sms, stream);
}

// Tiles of an item's stationary block.  Four 128-row tiles take the most out of every streamed tile, but a launch with
// few items then ends with one item per SM and the others idle; with two or one, each tile serves two or four
// accumulator slots and an item is a half or a quarter as long.  The time of the call's sweeps is estimated in us from the
// rounds of the items (one streamed tile against four accumulators) and what an item costs by itself: a launch takes its
// longest item, or an SM's mean load and a part of the shortest item.  Blocks of less than four tiles have to win by 5 %.
// The constants are a fit to 400 problems (1 to 1024 heads, 60 to 8192 tokens, batches of up to 64 sequences) timed with each
// block size: the choice is 0.4 % behind the best on average, 15 % at worst (heads of 200 tokens), and never slower than four
// tiles.  32 heads, 4 / 2 / 1 tiles: 1001 tokens 45 / 33 / 31 us, 2048 tokens 80 / 56 / 66, 4096 tokens 168 / 173 / 204; 8 heads,
// 3000 tokens 115 / 72 / 78; 1024 heads, 300 tokens 115 / 159 / 186; 256 heads, 12 sequences of 200 to 800 tokens 575 / 731 / 988.
int block_tiles(const Shape& s, const int32_t* cu_host, int n_sms, bool row_sweep) {
  constexpr float kRound[3] = {2.2f, 2.35f, 2.55f}, kItem[3] = {1.2f, 3.1f, 3.1f};
  constexpr float kShortest = 0.55f, kFixed = 3.5f, kCounter = 3.f, kMargin = 1.05f;
  constexpr float kShare[5] = {0.f, 0.25f, 0.5f, 1.f, 1.f};          // rounds per streamed tile of a block, by its tiles
  const float n_lh = (float)s.n_layers * s.Hq;
  int best = kQ;
  float best_cost = 0.f;
  for (int v = 0, tpb = kQ; tpb >= 1; ++v, tpb /= 2) {
    float cost = 0.f;
    for (int sweep = row_sweep ? 0 : 1; sweep < 2; ++sweep) {
      float sum = 0.f, longest = 0.f, shortest = 1e9f, items = 0.f;
      auto block = [&](float n_streamed, float share) {
        const float rounds = fmaxf(1.f, n_streamed * share);
        longest = fmaxf(longest, rounds);
        shortest = fminf(shortest, rounds);
        return rounds;
      };
      for (int i = 0; i < s.n_seqs; ++i) {
        const int n = (cu_host[i + 1] - cu_host[i] + kTile - 1) / kTile;
        const int full = n / tpb, q = n - full * tpb;                // full blocks, tiles of the last one
        if (full > 0) {                                              // from the least streamed tiles to the most
          const int most = !s.causal ? n : sweep == 0 ? full * tpb : n;
          const int least = !s.causal ? n : sweep == 0 ? tpb : n - (full - 1) * tpb;
          block((float)least, kShare[tpb]);
          block((float)most, kShare[tpb]);
          sum += 0.5f * full * (least + most) * kShare[tpb];
        }
        if (q > 0) sum += block(s.causal && sweep == 1 ? (float)q : (float)n, sweep == 1 && tpb == kQ ? 1.f : kShare[q]);
        items += full + (q > 0);
      }
      const float item = kItem[v], mean = (kRound[v] * sum + item * items) * n_lh / n_sms;
      longest = kRound[v] * longest + item;
      cost += kFixed + (items * n_lh <= n_sms ? longest : fmaxf(longest, mean + kShortest * (kRound[v] * shortest + item)));
      if (sweep == 1 && items * n_lh > 2 * n_sms) cost += kCounter;
    }
    if (tpb == kQ || cost < best_cost) { best = tpb; best_cost = tpb == kQ ? cost / kMargin : cost; }
  }
  return best;
}

}  // namespace

size_t score_tensor_counter_bytes() { return 256; }

int score_tensor_plan(const Shape& s, const TensorView& Q, const TensorView& K, ScoreTensorMaps* maps) {
  static_assert(sizeof(CUtensorMap) == sizeof(maps->q) && alignof(CUtensorMap) <= 64, "tensor map storage");
  if (Q.dtype != K.dtype || (Q.dtype != KVCRUSH_BF16 && Q.dtype != KVCRUSH_FP16)) return TENSOR_PLAN_NO;
  if (s.D < 8 || s.D > 128 || s.D % 8 != 0) return TENSOR_PLAN_NO;      // other widths ride in the 64- or 128-wide kernel
  if (s.T < 1) return TENSOR_PLAN_NO;
  if (encode_fn() == nullptr) return TENSOR_PLAN_NO_ENCODER;
  if (!make_map(reinterpret_cast<CUtensorMap*>(maps->q), Q, s.D, s.T, s.Hq, s.n_layers) ||
      !make_map(reinterpret_cast<CUtensorMap*>(maps->k), K, s.D, s.T, s.Hkv, s.n_layers))
    return TENSOR_PLAN_NO;                                               // strides or extents the TMA unit cannot take
  return TENSOR_PLAN_OK;
}


int launch_score_tensor(const Shape& s, const int32_t* cu_host, const TensorView& Q, const ScoreTensorMaps& maps,
                        float scale_log2, const float* lse_in, float lse_in_mul, float* lse2_ws,
                        int* counters, float* scores, float* lse_out, int normalize, int32_t* status,
                        const ScoreDiag& diag, cudaStream_t stream) {
  static_assert(sizeof(PAux) <= 26624, "aux block too large");
  if (!(scale_log2 > 0.f)) return KVCRUSH_ERR_UNSUPPORTED;
  const CUtensorMap& mq = *reinterpret_cast<const CUtensorMap*>(maps.q);
  const CUtensorMap& mk = *reinterpret_cast<const CUtensorMap*>(maps.k);
  const int n_sms = sm_count();
  PersistArgs a{};
  a.s = s; a.scale_log2 = scale_log2; a.normalize = normalize; a.bf16 = Q.dtype == KVCRUSH_BF16; a.status = status; a.scores = scores;
  const bool sw = diag.short_waits != 0;
  if (!lse_in && score_window_fits(s)) {
    const int rc = launch_score_window(s, cu_host, Q, maps, scale_log2, scores, lse_out, normalize, status, diag, stream);
    // no room for its clusters on this GPU: two sweeps (but not for a diagnostic call, which tests the kernel a call takes)
    if (rc != KVCRUSH_ERR_UNSUPPORTED || sw || diag.withhold_first_item) return rc;
  }
  a.withhold_first_item = diag.withhold_first_item;
  // Work items per (layer, head): every block of tpb 128-row tiles for the column sweep; for the row sweep only the
  // blocks that hold voting queries.
  auto count = [&](int tpb, bool row_sweep) {
    long long items = 0;
    for (int i = 0; i < s.n_seqs; ++i) {
      const int len = cu_host[i + 1] - cu_host[i], rows = tpb * kTile;
      items += (len + rows - 1) / rows - (row_sweep && s.window > 0 && len > s.window ? (len - s.window) / rows : 0);
    }
    return items;
  };
  a.n_lh = s.n_layers * s.Hq;
  const long long items_all = count(1, false);
  if (items_all == 0) return KVCRUSH_OK;
  if (items_all * a.n_lh > 0x7FFFFFFFLL) return KVCRUSH_ERR_UNSUPPORTED;
  // Tiles of the column sweep with queries that do not vote: behind a sequence's end, unless nothing is packed there, and before
  // a window.  Without any (single sequences, lengths that are multiples of 128) the sweep does without the edge warp.
  bool edge = false;
  for (int i = 0; i < s.n_seqs; ++i) {
    const int len = cu_host[i + 1] - cu_host[i];
    edge = edge || (len % kTile != 0 && cu_host[i + 1] < s.T) || (s.window > 0 && len > s.window && (len - s.window) % kTile != 0);
  }
  a.tpb = s.window > 0 ? kQ : block_tiles(s, cu_host, n_sms, !lse_in);
  bool zeroed = false;
  auto plan = [&](bool row_sweep, int* counter) {
    const long long items = count(a.tpb, row_sweep);
    a.max_blocks = (s.max_seqlen + a.tpb * kTile - 1) / (a.tpb * kTile);
    a.n_items = (int)items;
    a.total_items = (int)(items * a.n_lh);
    const long long tail = (4LL * n_sms + items - 1) / items;   // pairs whose items make up about four rounds of the grid
    a.tail_lh = (int)(tail < a.n_lh ? tail : a.n_lh);
    // Dealt out in advance only while a block gets two items at most: 6 % faster then (13 % with one), but up to 23 %
    // slower with three or four, where the snake meets loads that are no longer even (64 heads of 800, 200, 400 and 600
    // tokens: 79 us against 64).
    a.counter = a.tail_lh == a.n_lh && a.total_items <= 2 * n_sms ? nullptr : counter;
    if (a.counter && !zeroed) {
      if (cudaMemsetAsync(counters, 0, 2 * sizeof(int), stream) != cudaSuccess) return false;
      zeroed = true;
    }
    return true;
  };
  int rc;
  if (!lse_in) {
    if (!plan(true, counters)) return KVCRUSH_ERR_CUDA;
    a.lse2_out = lse2_ws; a.lse_nat_out = lse_out;
    // Sequences of one tile have nothing to split (4 layers x 32 heads x 64 of 64 tokens, both sweeps: 368 -> 302 us).
    rc = s.max_seqlen > kTile ? launch_persist<false, true>(mq, mk, a, edge, sw, n_sms, stream) : launch_persist<false, false>(mq, mk, a, edge, sw, n_sms, stream);
    if (rc != KVCRUSH_OK) return rc;
    a.lse = lse2_ws; a.lse_mul = 1.f;
  } else {
    a.lse = lse_in; a.lse_mul = lse_in_mul;
  }
  if (!plan(false, counters + 1)) return KVCRUSH_ERR_CUDA;
  // The column sweep need not wait for the whole row sweep where that is the launch before it.  It saves 3 to 5 us a call (32
  // heads over 8, 1001 tokens, whole pass 54.8 -> 50.0 us, with operands that no cache holds 55.8 -> 51.2; 32 heads of 4096 tokens
  // 192.3 -> 189.4), but this build of the kernel is 2 % slower in its loop (32 x 32 x 8192 tokens 20.0 -> 20.3 ms), so that only
  // calls of one or two items a block take it.
  if (!lse_in && !a.counter) return a.tpb < kQ ? launch_persist<true, true, true>(mq, mk, a, edge, sw, n_sms, stream) : launch_persist<true, false, true>(mq, mk, a, edge, sw, n_sms, stream);
  return a.tpb < kQ ? launch_persist<true, true>(mq, mk, a, edge, sw, n_sms, stream) : launch_persist<true, false>(mq, mk, a, edge, sw, n_sms, stream);
}

}  // namespace kvc

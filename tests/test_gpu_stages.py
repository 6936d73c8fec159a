"""GPU parity, stage by stage, through the C ABI: signature, selection and compaction are
bit-exact when fed the oracle's float32 scores; scores agree within 1e-5 + 2e-3*|oracle|."""
import numpy as np
import pytest

from oracle import kvcrush_oracle as O
from paper_2503_00022_b200 import inputs
import kvc_testlib as TL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_00022_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def _dev():
    import torch
    return torch.device("cuda:0")


# ---------------------------------------------------------------------------------------------
# signature + select on oracle scores
# ---------------------------------------------------------------------------------------------

def _select_case(B, Hq, Hkv, seqlens, budgets, n_layers, ties, mode, seed, sig_keep=None, share_importance=True):
    import torch
    dev = _dev()
    S, T = len(seqlens), int(sum(seqlens))
    cu = np.concatenate([[0], np.cumsum(seqlens)]).astype(np.int64)
    b_imp = np.asarray([b[0] for b in budgets], dtype=np.int32)
    b_rep = np.asarray([b[1] for b in budgets], dtype=np.int32)
    scores = np.zeros((n_layers, Hq, T), dtype=np.float32)
    for l in range(n_layers):
        for s, L in enumerate(seqlens):
            scores[l, :, cu[s]:cu[s + 1]] = inputs.random_scores(Hq, L, seed + 17 * l + s, tie_levels=ties)
    explicit = inputs.random_anchor_bits(Hq, seed + 5)
    w = inputs.Workload("t", n_layers, Hq, Hkv, 16, tuple(seqlens), inputs.FP32, inputs.FP32, 0.25)
    prob = B.Problem(n_layers, Hq, Hkv, 16, seqlens, device=dev)
    # share_importance: the signature stage writes the token importance and the selection stage takes it over;
    # without it the selection stage makes its own pass over the scores
    cp = B.CompressionPass(prob, b_imp[None, :], b_rep[None, :], sig_keep=sig_keep, anchor_mode=mode,
                           anchor_bits=explicit if mode == B.ANCHOR_EXPLICIT else None,
                           share_importance=share_importance)
    dscores = torch.from_numpy(scores).to(dev)
    for rep in range(2):                      # twice: results must not depend on leftover scratch
        cp.signature(dscores)
        cp.select(dscores)
        torch.cuda.synchronize()
        cp.check_status()
        sigs = cp.sigs.cpu().numpy().view(np.uint32)
        theta = cp.theta.cpu().numpy()
        np.testing.assert_array_equal(cp.n_kept.cpu().numpy(),        # the optional per-segment count output
                                      np.tile(np.minimum(b_imp + b_rep, np.asarray(seqlens)), (n_layers, 1)))
        for l in range(n_layers):
            ref = TL.oracle_select_layer(w, scores[l], b_imp, b_rep,
                                         None if sig_keep is None else np.asarray(sig_keep).reshape(-1),
                                         mode, explicit)
            for s in range(S):
                np.testing.assert_array_equal(theta[l, s], ref[s]["theta"])
                np.testing.assert_array_equal(sigs[l, cu[s]:cu[s + 1]], ref[s]["sig"])
                np.testing.assert_array_equal(cp.kept(l, s), ref[s]["idx"].astype(np.int32))
                seg = l * S + s
                kind = cp.kind[int(cp.cu_kept_host[seg]):int(cp.cu_kept_host[seg + 1])].cpu().numpy()
                np.testing.assert_array_equal(kind, ref[s]["kind"])


@pytest.mark.parametrize("Hq,Hkv,seqlens,budgets,ties,mode", [
    (8, 8, [512], [(64, 64)], 0, 0),
    (32, 32, [4096], [(512, 512)], 0, 0),
    (32, 8, [1000, 37, 2049], [(100, 150), (5, 4), (300, 212)], 0, 0),
    (32, 8, [1000, 333], [(100, 150), (40, 43)], 4, 0),            # heavy ties everywhere
    (40, 10, [777, 1025], [(64, 32), (100, 101)], 2, 1),           # two signature words, MEAN anchor
    (128, 16, [600], [(50, 70)], 0, 2),                            # four words, explicit (random) anchor
    (4, 1, [300, 300], [(0, 30), (30, 0)], 3, 0),                  # pure KVCrush / pure H2O
    (95, 95, [300], [(40, 30)], 0, 0),                             # a tile of scores just below, at and above 48 KB of
    (96, 96, [300], [(40, 30)], 0, 0),                             # shared memory
    (97, 97, [300], [(40, 30)], 0, 0),
    (16, 16, [100, 1, 64], [(60, 60), (1, 0), (3, 1)], 0, 1),      # budget >= length keeps all; L = 1
    (32, 32, [5000], [(10, 1)], 0, 0),                             # one huge bucket
    (32, 32, [2500], [(20, 2)], 2, 1),
])
def test_signature_and_select_bit_exact_on_oracle_scores(B, Hq, Hkv, seqlens, budgets, ties, mode):
    _select_case(B, Hq, Hkv, seqlens, budgets, 2, ties, mode, seed=100 + Hq + len(seqlens))


def test_select_long_sequence_32k(B):
    _select_case(B, 32, 8, [32768], [(3277, 3277)], 1, 0, 0, seed=9)
    _select_case(B, 32, 8, [32768], [(3277, 3277)], 1, 0, 0, seed=9, share_importance=False)


@pytest.mark.parametrize("Hq,Hkv,seqlens,budgets,ties,mode", [
    (32, 8, [1000, 37, 2049], [(100, 150), (5, 4), (300, 212)], 0, 0),
    (32, 8, [1000, 333], [(100, 150), (40, 43)], 4, 0),
    (40, 10, [777, 1025], [(64, 32), (100, 101)], 2, 1),
])
def test_select_computes_the_importance_itself_when_none_is_handed_over(B, Hq, Hkv, seqlens, budgets, ties, mode):
    _select_case(B, Hq, Hkv, seqlens, budgets, 2, ties, mode, seed=300 + Hq, share_importance=False)


def test_signature_thresholds_for_rows_beyond_the_register_kernel(B):
    """Rows longer than 32768 tokens take the streaming threshold kernel."""
    _select_case(B, 4, 2, [40000, 70], [(500, 300), (7, 9)], 1, 0, 0, seed=17)
    _select_case(B, 4, 2, [33000], [(100, 50)], 1, 3, 0, seed=18)


@pytest.mark.parametrize("Hq,L,b_imp,b_rep,ties", [
    (4, 13088, 900, 1300, 0), (4, 13216, 900, 1300, 0),      # a cluster of four blocks
    (128, 7488, 300, 1500, 0), (128, 7680, 300, 1500, 0),    # one block, the last segment staged whole and the first that is not
    (4, 33000, 2000, 3300, 0),                               # a cluster of eight: buckets of 10
    (4, 45000, 500, 9000, 0),                                # buckets of 5
    (4, 66000, 100, 300, 0),                                 # buckets of 220
    (4, 20000, 700, 1700, 3), (4, 300, 40, 60, 2),           # more than 256 candidates after the first round, ties cut
])
def test_select_at_the_edges_of_its_staging(B, Hq, L, b_imp, b_rep, ties):
    _select_case(B, Hq, Hq, [L], [(b_imp, b_rep)], 1, ties, 0, seed=330 + L % 97)


@pytest.mark.parametrize("Hq,L,n_short,b_imp,b_rep,ties,share", [
    (4, 13088, 32, 900, 1300, 0, True), (4, 13216, 32, 900, 1300, 0, True),     # the last segment staged whole, the first that is not
    (40, 12288, 32, 700, 1000, 0, True), (128, 9000, 32, 300, 1500, 2, True),   # two and four signature words
    (4, 20000, 32, 700, 1700, 3, False),                     # more than 256 candidates after the first round, ties cut
    (4, 33000, 64, 2000, 3300, 0, True),                     # signatures and 16-bit order in shared memory; buckets of 10
    (4, 45000, 64, 500, 9000, 0, False),                     # order in global memory; buckets of 5
    (4, 66000, 64, 100, 300, 2, True),                       # nothing staged, buckets of 220
])
def test_select_of_one_long_segment_among_many(B, Hq, L, n_short, b_imp, b_rep, ties, share):
    """One block a segment, because there are too many for clusters, and one of them too long to be staged whole."""
    seqlens = [L] + [33 + 7 * (i % 5) for i in range(n_short)]
    budgets = [(b_imp, b_rep)] + [(n // 6, n // 5) for n in seqlens[1:]]
    prob = B.Problem(1, Hq, Hq, 16, seqlens, device=_dev())
    assert B.lib().kvcrush_diag_select_blocks(prob.ref, 148, 8) == 1
    _select_case(B, Hq, Hq, seqlens, budgets, 1, ties, 0, seed=450 + L % 89, share_importance=share)


@pytest.mark.parametrize("Hq,seqlens,mode,ties", [
    (8, [1024, 1], 0, 0), (8, [1025, 40], 0, 0), (40, [1000, 33], 2, 1),          # 512 threads, 1024, 512
    (8, [300, 41, 1500] * 50, 0, 2), (72, [1025, 64] * 75, 2, 0),                 # more segments than SMs: 512
    (8, [70, 2, 260, 1] * 75, 2, 0), (8, [2048] + [33, 90] * 149, 0, 2),          # more than twice as many: 256
    (128, [2049] + [64, 20] * 149, 0, 0),                                         # 512 again
])
def test_select_in_blocks_of_every_size(B, Hq, seqlens, mode, ties):
    budgets = [(max(1, L // 6), L // 5) for L in seqlens]
    _select_case(B, Hq, Hq, seqlens, budgets, 1, ties, mode, seed=370 + len(seqlens))


@pytest.mark.parametrize("Hq,layers,seqlens,b_imp,b_rep,mode,ties,share", [
    (32, 1, [8192], 800, 1200, 0, 0, True), (8, 3, [8193, 31, 1], 900, 1300, 1, 0, True),    # four blocks; parts of 32 tokens and none
    (8, 1, [8200], 300, 3, 0, 0, True), (8, 1, [16385], 100, 1, 2, 0, True),                 # fewer buckets than blocks: order in global memory
    (128, 1, [9000], 400, 1700, 1, 0, True), (72, 2, [17001, 100], 0, 2900, 2, 2, False),    # four and three signature words; nothing important
    (32, 5, [8222], 500, 0, 0, 0, True), (40, 8, [8233], 333, 2222, 0, 3, True),             # no buckets; ties cut across blocks
    (4, 2, [20000], 700, 1700, 0, 2, False), (4, 1, [45000], 500, 9000, 0, 0, True),         # eight blocks
    (4, 32, [12300], 700, 900, 0, 0, True), (4, 33, [12300], 700, 900, 0, 0, True),          # as many segments as take clusters, and one more
])
def test_select_by_a_cluster_of_blocks(B, Hq, layers, seqlens, b_imp, b_rep, mode, ties, share):
    budgets = [(b_imp, b_rep)] + [(max(1, L // 6), L // 5) for L in seqlens[1:]]
    _select_case(B, Hq, Hq, seqlens, budgets, layers, ties, mode, seed=410 + Hq + layers, share_importance=share)


@pytest.mark.parametrize("seqlens,ties", [
    ([1, 2, 31, 32, 33, 256], 0), ([255, 256, 1, 100], 2),       # 8 keys a lane
    ([257, 31, 512], 0), ([511, 512, 480], 3),                   # 16
    ([513, 1023, 1024, 64] * 10, 0), ([1024, 700] * 19, 1),      # 32, more rows than the chip holds as blocks
    ([8193, 8192, 1], 0), ([16385, 40], 2), ([32767], 0),        # upper halves in shared memory; 2: more than 1024 in one bin
])
def test_thresholds_are_exact_for_every_row_kernel(B, seqlens, ties):
    budgets = [(max(1, L // 5), L // 7) for L in seqlens]
    _select_case(B, 32, 8, seqlens, budgets, 1, ties, 0, seed=230 + len(seqlens))


def test_signature_rank_other_than_budget_and_explicit_theta(B):
    import torch
    dev = _dev()
    _select_case(B, 16, 4, [400, 250], [(30, 30), (20, 21)], 1, 0, 0, seed=3, sig_keep=[[30, 20]])
    # explicit thresholds (the input form of Algorithm 1)
    Hq, L = 24, 333
    s = inputs.random_scores(Hq, L, 12)
    theta = np.linspace(0.05, 3.0, Hq).astype(np.float32)
    prob = B.Problem(1, Hq, Hq, 16, [L], device=dev)
    sigs = torch.empty((1, L, 1), dtype=torch.int32, device=dev)
    tout = torch.empty((1, 1, Hq), dtype=torch.float32, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_signature(prob, torch.from_numpy(s[None]).to(dev), sigs, theta_in=torch.from_numpy(theta).to(dev),
                        theta_out=tout, status=status)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(sigs.cpu().numpy().view(np.uint32)[0], O.signatures(s, theta))
    np.testing.assert_array_equal(tout.cpu().numpy().reshape(-1), theta)


# ---------------------------------------------------------------------------------------------
# compaction
# ---------------------------------------------------------------------------------------------

@pytest.mark.parametrize("dtype,D,Hkv,layout", [
    (inputs.FP16, 128, 8, "thd"), (inputs.BF16, 128, 4, "htd"), (inputs.FP32, 64, 8, "thd"), (inputs.BF16, 64, 3, "thd"),
])
def test_compact_bytes_equal_oracle(B, dtype, D, Hkv, layout):
    import torch
    dev = _dev()
    seqlens, n_layers = [300, 45, 1000], 3
    w = inputs.Workload("c", n_layers, Hkv, Hkv, D, tuple(seqlens), dtype, dtype, 0.25, base_seed=77)
    lis, _, _, kc, vc = TL.stack_layers(w, range(n_layers))
    g = np.random.Generator(np.random.Philox(5))
    budgets = np.asarray([[g.integers(1, L + 1) for L in seqlens] for _ in range(n_layers)], dtype=np.int32)
    prob = B.Problem(n_layers, Hkv, Hkv, D, seqlens, device=dev)
    tdt = {inputs.FP16: torch.float16, inputs.BF16: torch.bfloat16, inputs.FP32: torch.float32}[dtype]
    cp = B.CompressionPass(prob, budgets, np.zeros_like(budgets), cache_dtype=tdt)
    cu = w.cu_seqlens
    idx_host, ref_k, ref_v = [], [], []
    for l in range(n_layers):
        rk, rv = [], []
        for s, L in enumerate(seqlens):
            idx = np.sort(g.choice(L, size=int(budgets[l, s]), replace=False))
            idx_host.append(idx)
            rk.append(O.compact(kc[l, cu[s]:cu[s + 1]], idx))
            rv.append(O.compact(vc[l, cu[s]:cu[s + 1]], idx))
        ref_k.append(np.concatenate(rk))
        ref_v.append(np.concatenate(rv))
    cp.idx.copy_(torch.from_numpy(np.concatenate(idx_host).astype(np.int32)).to(dev))
    dk, dv = TL.torch_storage(kc, dtype, dev), TL.torch_storage(vc, dtype, dev)
    if layout == "htd":      # cache stored [layer, head, token, D]; the ABI sees it through strides
        dk = dk.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
        dv = dv.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    cp.k_out.fill_(0)
    cp.v_out.fill_(0)
    cp.compact(dk, dv)
    torch.cuda.synchronize()
    for l in range(n_layers):
        n = ref_k[l].shape[0]
        got_k = cp.k_out[l, :n].contiguous().view(torch.uint8).cpu().numpy()
        got_v = cp.v_out[l, :n].contiguous().view(torch.uint8).cpu().numpy()
        assert got_k.tobytes() == ref_k[l].tobytes()
        assert got_v.tobytes() == ref_v[l].tobytes()
        rest = cp.k_out[l, n:].contiguous().view(torch.uint8)
        assert int(rest.max()) == 0 if rest.numel() else True       # nothing written past the kept rows


# ---------------------------------------------------------------------------------------------
# scores
# ---------------------------------------------------------------------------------------------

def _score_case(B, w, impl, n_layers=None):
    import torch
    dev = _dev()
    layers = range(w.n_layers if n_layers is None else n_layers)
    lis, q, k, _, _ = TL.stack_layers(w, layers, with_cache=False)
    prob = B.Problem(len(lis), w.n_q_heads, w.n_kv_heads, w.head_dim, w.seqlens, causal=w.causal, device=dev)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    T = w.total_tokens
    scores = torch.full((len(lis), w.n_q_heads, T), -1.0, dtype=torch.float32, device=dev)
    lse = torch.empty_like(scores)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_score(prob, dq, dk, scores, lse_out=lse, impl=impl, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0, status.cpu().tolist()
    g, gl = scores.cpu().numpy(), lse.cpu().numpy()
    oracle_c, oracle_lse = [], []
    for i, li in enumerate(lis):
        c, ol = TL.oracle_scores_layer(w, li)
        ok = TL.within_score_tolerance(g[i], c)
        assert ok.all(), (w.name, i, np.argwhere(~ok)[:5], g[i][~ok][:5], c[~ok][:5])
        np.testing.assert_allclose(gl[i], ol, rtol=0, atol=2e-4)
        oracle_c.append(c)
        oracle_lse.append(ol)
    # the row log-sum-exp as a prefill kernel would hand it over - here the ORACLE's, rounded to float32, so that
    # nothing of the library's first sweep is involved: the second sweep alone must reproduce the oracle's column sums
    lse_o = torch.from_numpy(np.stack(oracle_lse).astype(np.float32)).to(dev)
    scores3 = torch.full_like(scores, -1.0)
    B.kvcrush_score(prob, dq, dk, scores3, lse_in=lse_o, impl=impl, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    g3 = scores3.cpu().numpy()
    for i, c in enumerate(oracle_c):
        ok = TL.within_score_tolerance(g3[i], c)
        assert ok.all(), (w.name, "oracle lse", i, np.argwhere(~ok)[:5], g3[i][~ok][:5], c[~ok][:5])
    # supplying the row log-sum-exp skips the first sweep and gives the same scores
    scores2 = torch.empty_like(scores)
    B.kvcrush_score(prob, dq, dk, scores2, lse_in=lse, impl=impl, workspace=ws, status=status)
    torch.cuda.synchronize()
    np.testing.assert_allclose(scores2.cpu().numpy(), g, rtol=1e-4, atol=1e-6)
    # normalize = the paper's 1/S
    B.kvcrush_score(prob, dq, dk, scores2, normalize=True, impl=impl, workspace=ws, status=status)
    torch.cuda.synchronize()
    cu = w.cu_seqlens
    n2 = scores2.cpu().numpy()
    for s, L in enumerate(w.seqlens):
        np.testing.assert_allclose(n2[:, :, cu[s]:cu[s + 1]] * L, g[:, :, cu[s]:cu[s + 1]], rtol=1e-5, atol=1e-7)
    return g


SIMT_CASES = [
    inputs.Workload("simt_cfg1", 1, 8, 8, 64, (512,), inputs.FP32, inputs.FP32, 0.25, base_seed=1100),
    inputs.Workload("simt_ragged_gqa", 2, 8, 2, 32, (130, 1, 257), inputs.BF16, inputs.BF16, 0.25, base_seed=21),
    inputs.Workload("simt_noncausal", 1, 4, 4, 128, (200, 96), inputs.BF16, inputs.BF16, 0.25, base_seed=22, causal=False),
]


@pytest.mark.parametrize("w", SIMT_CASES, ids=lambda w: w.name)
def test_score_simt_matches_oracle(B, w):
    _score_case(B, w, B.SCORE_SIMT)


TENSOR_CASES = [
    inputs.Workload("tc_one_tile", 1, 2, 2, 128, (128,), inputs.BF16, inputs.BF16, 0.25, base_seed=31),
    inputs.Workload("tc_ragged_tail", 1, 4, 4, 128, (700,), inputs.BF16, inputs.BF16, 0.25, base_seed=32),
    inputs.Workload("tc_gqa_varlen", 2, 8, 2, 128, (300, 1, 129, 1000), inputs.BF16, inputs.BF16, 0.25, base_seed=33),
    inputs.Workload("tc_d64", 1, 4, 2, 64, (513, 64), inputs.BF16, inputs.BF16, 0.25, base_seed=34),
    inputs.Workload("tc_noncausal", 1, 4, 4, 128, (333, 260), inputs.BF16, inputs.BF16, 0.25, base_seed=35, causal=False),
    inputs.Workload("tc_2k", 1, 8, 8, 128, (2048,), inputs.BF16, inputs.BF16, 0.25, base_seed=36),
    # more sequences than one warp decodes at once, lengths around every tile / block boundary, an empty sequence
    inputs.Workload("tc_many_seqs", 1, 2, 1, 64, tuple([127, 128, 129, 255, 256, 257, 0, 1, 383, 384, 385, 512] * 3 + [40, 300]),
                    inputs.BF16, inputs.BF16, 0.25, base_seed=37),
    inputs.Workload("tc_128_heads", 1, 128, 16, 64, (260,), inputs.BF16, inputs.BF16, 0.25, base_seed=38),
]


@pytest.mark.parametrize("w", TENSOR_CASES, ids=lambda w: w.name)
def test_score_tensor_matches_oracle(B, w):
    g = _score_case(B, w, B.SCORE_TENSOR)
    # the CUDA-core kernels see the same inputs: the two device paths agree far inside the tolerance
    import torch
    dev = _dev()
    lis, q, k, _, _ = TL.stack_layers(w, range(w.n_layers), with_cache=False)
    prob = B.Problem(w.n_layers, w.n_q_heads, w.n_kv_heads, w.head_dim, w.seqlens, causal=w.causal, device=dev)
    scores = torch.empty((w.n_layers, w.n_q_heads, w.total_tokens), dtype=torch.float32, device=dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_score(prob, TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev), scores,
                    impl=B.SCORE_SIMT, workspace=ws, status=status)
    torch.cuda.synchronize()
    np.testing.assert_allclose(g, scores.cpu().numpy(), rtol=2e-4, atol=1e-6)


@pytest.mark.parametrize("layers,Hq,Hkv,D,seqlens,causal", [
    (16, 32, 8, 64, (513, 640, 768, 897, 1), True),            # four tiles a block; last blocks of 1, 1, 2 and 4 tiles
    (16, 32, 32, 64, (1100, 300), False),                      # the same without a mask
    (1, 32, 8, 128, (2048,), True),                            # two tiles a block
    (1, 32, 8, 128, (1700, 130), True),                        # two, last blocks of 2 tiles with one short
    (2, 16, 4, 64, (1921,), False),
    (1, 32, 8, 128, (897,), True),                             # one tile a block, four slots each
    (1, 8, 8, 64, (5000,), True),                              # one, more items than SMs dealt out in advance
])
def test_scores_with_every_block_size(B, layers, Hq, Hkv, D, seqlens, causal):
    """Blocks of 4, 2 and 1 stationary tiles and their partial last blocks: the CUDA-core kernels on the same inputs agree
    within the score tolerance's tenth, the oracle on two heads within the tolerance."""
    import torch
    dev = _dev()
    w = inputs.Workload("blk", layers, Hq, Hkv, D, seqlens, inputs.BF16, inputs.BF16, 0.25, base_seed=250 + D, causal=causal)
    lis, q, k, _, _ = TL.stack_layers(w, range(layers), with_cache=False)
    prob = B.Problem(layers, Hq, Hkv, D, seqlens, causal=causal, device=dev)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    got = {}
    for impl in (B.SCORE_TENSOR, B.SCORE_SIMT):
        sc, ls = (torch.full((layers, Hq, w.total_tokens), -1.0, dtype=torch.float32, device=dev) for _ in range(2))
        B.kvcrush_score(prob, dq, dk, sc, lse_out=ls, impl=impl, workspace=ws, status=status)
        got[impl] = (sc.cpu().numpy(), ls.cpu().numpy())
    assert status.cpu().tolist()[0] == 0
    np.testing.assert_allclose(got[B.SCORE_TENSOR][0], got[B.SCORE_SIMT][0], rtol=2e-4, atol=1e-6)
    np.testing.assert_allclose(got[B.SCORE_TENSOR][1], got[B.SCORE_SIMT][1], rtol=0, atol=2e-4)
    cu, G = w.cu_seqlens, Hq // Hkv
    for s, L in enumerate(seqlens):
        a, b = int(cu[s]), int(cu[s + 1])
        for h in (0, Hq - 1):
            c, _ = O.scores(inputs.widen(lis[-1].q[a:b, h:h + 1], w.qk_dtype),
                            inputs.widen(lis[-1].k[a:b, h // G:h // G + 1], w.qk_dtype), causal)
            assert TL.within_score_tolerance(got[B.SCORE_TENSOR][0][-1, h:h + 1, a:b], c).all(), (s, h)


def test_score_tensor_rejects_fp32_and_auto_falls_back_to_cuda_cores(B):
    import torch
    dev = _dev()
    w = SIMT_CASES[0]
    lis, q, k, _, _ = TL.stack_layers(w, range(1), with_cache=False)
    prob = B.Problem(1, w.n_q_heads, w.n_kv_heads, w.head_dim, w.seqlens, device=dev)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    scores = torch.empty((1, w.n_q_heads, w.total_tokens), dtype=torch.float32, device=dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    with pytest.raises(B.KvcrushError) as e:
        B.kvcrush_score(prob, dq, dk, scores, impl=B.SCORE_TENSOR, workspace=ws, status=status)
    assert e.value.code == B.ERR_UNSUPPORTED
    B.kvcrush_score(prob, dq, dk, scores, impl=B.SCORE_AUTO, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert torch.isfinite(scores).all()


@pytest.mark.parametrize("impl_name", ["SCORE_TENSOR", "SCORE_SIMT"])
def test_score_head_major_layout_and_explicit_scale(B, impl_name):
    """Q/K stored [layer, head, token, D] (reached through strides) and a caller-chosen softmax scale."""
    import torch
    dev = _dev()
    impl = getattr(B, impl_name)
    w = inputs.Workload("hm", 2, 4, 2, 128, (391, 130), inputs.BF16, inputs.BF16, 0.25, base_seed=41)
    lis, q, k, _, _ = TL.stack_layers(w, range(2), with_cache=False)
    scale = 0.05
    prob = B.Problem(2, 4, 2, 128, w.seqlens, causal=True, softmax_scale=scale, device=dev)
    dq = TL.torch_storage(q, w.qk_dtype, dev).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    dk = TL.torch_storage(k, w.qk_dtype, dev).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    assert dq.stride(1) == 128 and dq.stride(2) == 128 * w.total_tokens
    scores = torch.empty((2, 4, w.total_tokens), dtype=torch.float32, device=dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_score(prob, dq, dk, scores, impl=impl, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    g = scores.cpu().numpy()
    cu = w.cu_seqlens
    for l, li in enumerate(lis):
        for s_, L in enumerate(w.seqlens):
            a, b = int(cu[s_]), int(cu[s_ + 1])
            c, _ = O.scores(inputs.widen(li.q[a:b], w.qk_dtype), inputs.widen(li.k[a:b], w.qk_dtype), True, scale=scale)
            assert TL.within_score_tolerance(g[l][:, a:b], c).all()


def test_score_leaves_at_once_when_status_already_flags_an_error(B):
    """The tensor-core kernels read the status word first: a launch that follows a reported device error does
    no work (outputs untouched) and keeps the first error's record."""
    import torch
    dev = _dev()
    w = TENSOR_CASES[1]
    lis, q, k, _, _ = TL.stack_layers(w, range(1), with_cache=False)
    prob = B.Problem(1, w.n_q_heads, w.n_kv_heads, w.head_dim, w.seqlens, device=dev)
    scores = torch.full((1, w.n_q_heads, w.total_tokens), -5.0, dtype=torch.float32, device=dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.tensor([B.DEV_TIMEOUT, 2, 17, 0], dtype=torch.int32, device=dev)
    B.kvcrush_score(prob, TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev), scores,
                    impl=B.SCORE_TENSOR, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist() == [B.DEV_TIMEOUT, 2, 17, 0]
    assert bool((scores == -5.0).all())
    status.zero_()                                           # and the same call works once the word is cleared
    B.kvcrush_score(prob, TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev), scores,
                    impl=B.SCORE_TENSOR, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0 and bool((scores >= 0).all())


def test_a_bounded_wait_that_runs_out_is_reported_and_the_context_stays_usable(B):
    """Every barrier wait of the tensor-core kernels is bounded.  Here one is made to run out, on the smallest problem
    there is (one work item, one thread block): through the library's diagnostic entry point (exported, not part of
    the public header) the producer warp fetches its work item and then stops before announcing it and before issuing
    any copy, and the kernels run in their instantiation with a short poll limit.  Nothing is in flight, so the
    consumers' first waits expire, the block flags the status word, frees its tensor memory and the kernel returns
    normally; the second sweep, enqueued by the same call, waits for the first, finds the status word set and leaves.  The outputs
    stay untouched, and the same problem goes through the public entry point once the word is cleared."""
    import ctypes
    import torch
    dev = _dev()
    lib = B.lib()
    fn = lib.kvcrush_diag_score
    vp, i32 = ctypes.c_void_p, ctypes.c_int
    fn.restype = i32
    fn.argtypes = [ctypes.POINTER(B.ProblemStruct), ctypes.POINTER(B.TensorStruct), ctypes.POINTER(B.TensorStruct),
                   vp, vp, vp, i32, i32, vp, ctypes.c_size_t, vp, vp, i32, i32]
    w = inputs.Workload("one_item", 1, 1, 1, 128, (128,), inputs.BF16, inputs.BF16, 0.25, base_seed=55)
    lis, q, k, _, _ = TL.stack_layers(w, range(1), with_cache=False)
    prob = B.Problem(1, 1, 1, 128, w.seqlens, device=dev)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    qs, ks = B.tensor_struct(dq), B.tensor_struct(dk)
    scores = torch.full((1, 1, 128), -5.0, dtype=torch.float32, device=dev)
    lse = torch.full((1, 1, 128), -7.0, dtype=torch.float32, device=dev)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    stream = int(torch.cuda.current_stream().cuda_stream)
    rc = fn(prob.ref, ctypes.byref(qs), ctypes.byref(ks), None, scores.data_ptr(), lse.data_ptr(), 0, B.SCORE_TENSOR,
            ws.data_ptr(), ws.numel(), status.data_ptr(), stream, 1, 1)
    assert rc == B.OK
    torch.cuda.synchronize()                                 # the kernels came back by themselves
    st = status.cpu().tolist()
    assert st[0] == B.DEV_TIMEOUT and st[1] == 1 and st[2] == 0, st          # kernel id 1: the row sweep; block 0
    assert bool((scores == -5.0).all()) and bool((lse == -7.0).all())
    # the public entry point gives the oracle's scores on the same context once the word is cleared
    status.zero_()
    scores.fill_(-5.0)
    B.kvcrush_score(prob, dq, dk, scores, lse_out=lse, impl=B.SCORE_TENSOR, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    c, ol = TL.oracle_scores_layer(w, lis[0])
    assert TL.within_score_tolerance(scores.cpu().numpy()[0], c).all()
    np.testing.assert_allclose(lse.cpu().numpy()[0], ol, rtol=0, atol=2e-4)


def test_no_kernel_starts_beside_a_row_sweep_whose_first_block_gave_up(B):
    """The first block of the row sweep gives up (see above) while the others are in the middle of long items.  The column
    sweep of the same call is set up meanwhile, block after block on SMs that become free, finds the status word set and
    leaves; the kernel after the call must find every row log-sum-exp of the others written all the same."""
    import ctypes
    import torch
    dev = _dev()
    fn = B.lib().kvcrush_diag_score
    vp, i32 = ctypes.c_void_p, ctypes.c_int
    fn.restype = i32
    fn.argtypes = [ctypes.POINTER(B.ProblemStruct), ctypes.POINTER(B.TensorStruct), ctypes.POINTER(B.TensorStruct),
                   vp, vp, vp, i32, i32, vp, ctypes.c_size_t, vp, vp, i32, i32]
    Hq, L = 1, 75776                                         # 296 blocks of 256 rows, two for each SM: about 0.7 ms, a limit 0.3
    g = torch.Generator(device=dev).manual_seed(12)
    q, k = (torch.randn((1, L, Hq, 64), generator=g, device=dev).to(torch.bfloat16) for _ in range(2))
    prob = B.Problem(1, Hq, Hq, 64, (L,), device=dev)
    qs, ks = B.tensor_struct(q), B.tensor_struct(k)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    scores = torch.full((1, Hq, L), -5.0, device=dev)
    lse, seen = torch.full_like(scores, -7.0), torch.empty_like(scores)
    status, status2 = (torch.zeros(4, dtype=torch.int32, device=dev) for _ in range(2))
    stream = int(torch.cuda.current_stream().cuda_stream)
    assert fn(prob.ref, ctypes.byref(qs), ctypes.byref(ks), None, scores.data_ptr(), lse.data_ptr(), 0, B.SCORE_TENSOR,
              ws.data_ptr(), ws.numel(), status.data_ptr(), stream, 1, 2) == B.OK
    B.kvcrush_pool_scores(prob, lse, 1, seen, status=status2, stream=stream)      # a copy by a kernel of the library
    torch.cuda.synchronize()
    assert status.tolist()[:3] == [B.DEV_TIMEOUT, 1, 0]
    written = lse != -7.0
    assert 0.5 < written.float().mean().item() < 1.0                     # the first block's items are missing
    assert torch.equal(seen, lse)
    status.zero_()
    B.kvcrush_score(prob, q, k, scores, lse_out=seen, impl=B.SCORE_TENSOR, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.tolist()[0] == 0 and torch.equal(seen[written], lse[written])


@pytest.mark.parametrize("stage,small,large", [("signature", 9000, 32000), ("decode", 24000, 40000), ("simt", 128, 256)])
def test_threads_with_different_sizes_do_not_take_each_others_launches_away(B, stage, small, large):
    """Two threads issue calls whose kernels take different amounts of dynamic shared memory, on streams of their own, by raw
    calls and with a short interpreter switch interval, so that they meet between setting the kernel's limit and launching."""
    import ctypes
    import sys
    import threading
    import torch
    dev, lib = _dev(), B.lib()

    def job(n):
        stream, status = torch.cuda.Stream(), torch.zeros(4, dtype=torch.int32, device=dev)
        tail = (status.data_ptr(), ctypes.c_void_p(stream.cuda_stream))
        if stage == "signature":
            prob = B.Problem(1, 1, 1, 16, [n], device=dev)
            bufs = (torch.rand((1, 1, n), device=dev), torch.tensor([[n // 4]], dtype=torch.int32, device=dev),
                    torch.empty((1, n, 1), dtype=torch.int32, device=dev), torch.empty((1, 1, 1), device=dev))
            sc, keep, sigs, theta = (x.data_ptr() for x in bufs)
            fn, args = lib.kvcrush_signature, (prob.ref, sc, keep, None, sigs, theta, None, None, 0, *tail)
        elif stage == "decode":
            prob = B.Problem(1, 8, 1, 64, [n], device=dev)
            bufs = (torch.ones((1, 1, 8, 64), dtype=torch.bfloat16, device=dev), torch.ones((1, n, 1, 64), dtype=torch.bfloat16, device=dev),
                    torch.zeros((1, 8, n), device=dev))
            views = B.tensor_struct(bufs[0]), B.tensor_struct(bufs[1])
            fn, args = lib.kvcrush_score_decode, (prob.ref, *map(ctypes.byref, views), bufs[2].data_ptr(), *tail)
        else:
            prob = B.Problem(1, 1, 1, n, [64], device=dev)
            bufs = (torch.ones((1, 64, 1, n), device=dev), torch.empty((1, 1, 64), device=dev),
                    torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev))
            view = B.tensor_struct(bufs[0])
            fn, args = lib.kvcrush_score, (prob.ref, ctypes.byref(view), ctypes.byref(view), None, bufs[1].data_ptr(), None, 0,
                                           B.SCORE_SIMT, bufs[2].data_ptr(), bufs[2].numel(), *tail)
        return lambda: fn(*args), (prob, bufs, status, stream)

    jobs = [job(small), job(large)]
    assert all(call() == B.OK for call, _ in jobs)
    torch.cuda.synchronize()
    failed = []
    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        threads = [threading.Thread(target=lambda c=call: failed.append(sum(c() != B.OK for _ in range(20000)))) for call, _ in jobs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(interval)
    torch.cuda.synchronize()
    assert failed == [0, 0]


def test_pass_replays_from_a_cuda_graph(B):
    """The four stages enqueue kernels and one memset only, so a pass can be recorded once and replayed on new
    contents of the same tensors; the replayed result equals a direct run."""
    import torch
    dev = torch.device("cuda:0")
    w = inputs.Workload("graph", 2, 8, 2, 128, (600, 259), inputs.BF16, inputs.FP16, 0.25, base_seed=81)
    lis, q, k, kc, vc = TL.stack_layers(w, range(2))
    prob = B.Problem(2, 8, 2, 128, w.seqlens, device=dev)
    b_imp, b_rep = w.budgets()
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    dkc, dvc = TL.torch_storage(kc, w.cache_dtype, dev), TL.torch_storage(vc, w.cache_dtype, dev)
    direct = B.CompressionPass(prob, b_imp[None], b_rep[None], cache_dtype=torch.float16)
    direct.run(dq, dk, dkc, dvc)
    torch.cuda.synchronize()
    want = (direct.idx.clone(), direct.k_out.clone(), direct.scores.clone())
    cp = B.CompressionPass(prob, b_imp[None], b_rep[None], cache_dtype=torch.float16)
    zq, zk = torch.zeros_like(dq), torch.zeros_like(dk)
    cp.capture(zq, zk, dkc, dvc)                     # recorded on other contents
    zq.copy_(dq)
    zk.copy_(dk)
    for _ in range(2):
        cp.replay()
    torch.cuda.synchronize()
    cp.check_status()
    assert torch.equal(cp.idx, want[0]) and torch.equal(cp.k_out, want[1]) and torch.equal(cp.scores, want[2])


@pytest.mark.parametrize("dtype,D,Hq,Hkv,seqlens,causal,window", [
    (inputs.FP32, 64, 2, 1, (63, 64, 65), True, 0),          # around one tile of 64 rows
    (inputs.FP32, 8, 1, 1, (1,), True, 0),                   # the smallest problem
    (inputs.FP32, 64, 2, 1, (15, 0, 16, 1), True, 0),        # a logit a thread: no sequence above 16 tokens
    (inputs.FP32, 40, 2, 2, (16, 31, 17, 32), False, 0),     # 2 x 2 logits a thread: none above 32
    (inputs.FP32, 64, 1, 1, (30, 16, 33), True, 10),
    (inputs.FP32, 128, 1, 1, (1025,), True, 0),              # streamed tiles shared by 8 blocks, last tile of one row
    (inputs.FP32, 72, 4, 2, (190, 0, 129), False, 0),        # channels not a multiple of the shared-memory bank count
    (inputs.FP32, 256, 2, 2, (200,), True, 70),              # widest heads, window that cuts a tile
    (inputs.BF16, 200, 2, 1, (257,), True, 0),               # bf16 too wide for the tensor-core kernels
])
def test_cuda_core_scores_at_the_edges_of_their_tiles(B, dtype, D, Hq, Hkv, seqlens, causal, window):
    """fp32 sums of at most 1025 terms and an exponential of 2 ulp: far inside the score tolerance."""
    import torch
    dev = torch.device("cuda:0")
    w = inputs.Workload("simt", 2, Hq, Hkv, D, seqlens, dtype, dtype, 0.25, base_seed=190 + D, causal=causal)
    lis, q, k, _, _ = TL.stack_layers(w, range(2), with_cache=False)
    prob = B.Problem(2, Hq, Hkv, D, seqlens, causal=causal, device=dev, query_window=window)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    scores = torch.full((2, Hq, w.total_tokens), -1.0, device=dev)
    lse = torch.full_like(scores, 7.0)
    B.kvcrush_score(prob, TL.torch_storage(q, dtype, dev), TL.torch_storage(k, dtype, dev), scores, lse_out=lse,
                    impl=B.SCORE_SIMT, workspace=ws, status=status)
    g, gl = scores.cpu().numpy(), lse.cpu().numpy()
    assert status.cpu().tolist()[0] == 0
    cu = w.cu_seqlens
    for l, li in enumerate(lis):
        for s, L in enumerate(seqlens):
            a, b = int(cu[s]), int(cu[s + 1])
            if L == 0:
                continue
            j0 = max(0, L - window) if window else 0
            c, ol = O.scores(inputs.widen(li.q[a:b], dtype), inputs.widen(li.k[a:b], dtype), causal, rows=(j0, L))
            assert TL.within_score_tolerance(g[l][:, a:b], c).all(), (l, s)
            np.testing.assert_allclose(gl[l][:, a + j0:b], ol[:, j0:], rtol=0, atol=2e-5)
            assert (gl[l][:, a:a + j0] == 7.0).all()                       # rows that do not vote are not written


@pytest.mark.parametrize("layers,Hq,Hkv,D,seqlens,dtype", [
    (1, 8, 8, 64, [512], "float32"), (2, 4, 2, 32, [130, 1, 257], "float32"),               # CUDA cores, with and without clusters
    (1, 32, 8, 128, [1001], "bfloat16"), (1, 16, 16, 64, [300, 128, 700], "float16"),       # tensor cores, items dealt out in advance
    (2, 32, 8, 96, [1500, 1100], "bfloat16"),                                               # by the counter
])
def test_a_pass_follows_inputs_written_just_before_it(B, layers, Hq, Hkv, D, seqlens, dtype):
    """A whole pass right behind copies into its inputs gives what it gives after a synchronisation, bit for bit, also while the
    caches hold the old inputs.  (Its column sweep and its packing read before they wait, each behind a kernel of the same pass.
    The copies let nothing start early; launches that do come before the packing in the next test.)"""
    import torch
    dev, dt = _dev(), getattr(torch, dtype)
    T = sum(seqlens)
    prob = B.Problem(layers, Hq, Hkv, D, seqlens, device=dev)
    keep = np.asarray([[max(1, L // 8) for L in seqlens]], dtype=np.int32)
    cp = B.CompressionPass(prob, keep, keep, cache_dtype=dt)
    g = torch.Generator(device=dev).manual_seed(11)
    new = lambda h: torch.randn((layers, T, h, D), generator=g, device=dev).to(dt)
    q, k, v = new(Hq), new(Hkv), new(Hkv)
    outs = lambda: [x.clone() for x in (cp.scores, cp.theta, cp.sigs, cp.importance, cp.idx, cp.k_out, cp.v_out)]
    for _ in range(4):
        q2, k2 = new(Hq), new(Hkv)
        cp.run(q, k, k, v)                       # the old inputs are in every cache
        q.copy_(q2)
        k.copy_(k2)
        cp.run(q, k, k, v)
        got = outs()
        torch.cuda.synchronize()
        cp.run(q, k, k, v)
        torch.cuda.synchronize()
        cp.check_status()
        for a, b in zip(got, outs()):
            assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


@pytest.mark.parametrize("writer", ["decode", "pool", "gather"])
@pytest.mark.parametrize("layers,Hq,seqlens", [
    (1, 32, [1001]), (2, 8, [130, 1, 257, 30, 7, 90]),       # tokens no multiple of 4; several sequences in 128 tokens
    (3, 8, [8192]), (1, 4, [33000]), (20, 32, [700, 900]),   # every kernel of the thresholds
])
def test_signatures_follow_scores_written_by_the_launch_before(B, writer, layers, Hq, seqlens):
    """Scores written by a kernel that lets the thresholds' kernel be set up early, which does the same for the packing: that reads
    the scores before it waits.  Bit for bit what the same calls give with a synchronisation after each."""
    import torch
    dev = _dev()
    g = torch.Generator(device=dev).manual_seed(13)
    T, D = sum(seqlens), 64
    prob = B.Problem(layers, Hq, Hq, D, seqlens, device=dev)
    keep = np.asarray([[max(1, L // 8) for L in seqlens]], dtype=np.int32)
    cp = B.CompressionPass(prob, keep, keep)
    scores = torch.zeros((layers, Hq, T), device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    if writer == "decode":
        q = torch.randn((layers, len(seqlens), Hq, D), generator=g, device=dev).to(torch.bfloat16)
        k = torch.randn((layers, T, Hq, D), generator=g, device=dev).to(torch.bfloat16)
        write = lambda x: (scores.copy_(x), B.kvcrush_score_decode(prob, q, k, scores, status=status))
        source = lambda: torch.rand((layers, Hq, T), generator=g, device=dev)
    elif writer == "pool":
        write = lambda x: B.kvcrush_pool_scores(prob, x, 5, scores, status=status)
        source = lambda: torch.rand((layers, Hq, T), generator=g, device=dev)
    else:                                                    # every other token of a cache of twice the lengths
        before = B.Problem(layers, Hq, Hq, D, [2 * L for L in seqlens], device=dev)
        idx = torch.cat([2 * torch.arange(L, dtype=torch.int32, device=dev) for L in seqlens]).repeat(layers)
        cu_kept = torch.tensor(np.concatenate([[0], np.cumsum(list(seqlens) * layers)]), dtype=torch.int32, device=dev)
        write = lambda x: B.kvcrush_compact_scores(before, x, 0, cu_kept, idx, layers * T, scores, status=status)
        source = lambda: torch.rand((layers, Hq, 2 * T), generator=g, device=dev)

    def outputs(x, wait):
        for call in (lambda: write(x), lambda: cp.signature(scores), lambda: cp.select(scores)):
            call()
            if wait:
                torch.cuda.synchronize()
        return [t.clone() for t in (cp.theta, cp.sigs, cp.importance, cp.idx)]

    for _ in range(4):
        old, new = source(), source()
        outputs(old, False)                                  # the old scores are in every cache
        got = outputs(new, False)
        outputs(old, True)
        for a, b in zip(got, outputs(new, True)):
            assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
    cp.check_status()
    assert status.tolist()[0] == 0

"""GPU parity of the SnapKV-style importance pieces (Sec. 2.3 / 4.1.1 of the paper name them: an observation
window of the final prompt tokens, max pooling over neighbouring scores, the window itself kept):
windowed scores within 1e-5 + 2e-3*|oracle|, pooling and selection bit-exact."""
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


CASES = [
    # (workload, window)
    (inputs.Workload("win_tc_1k", 1, 4, 2, 128, (1000,), inputs.BF16, inputs.BF16, 0.25, base_seed=61), 64),
    (inputs.Workload("win_tc_ragged", 2, 4, 4, 128, (700, 31, 257, 1300), inputs.BF16, inputs.BF16, 0.25, base_seed=62), 200),
    (inputs.Workload("win_tc_d64", 1, 2, 1, 64, (513, 900), inputs.BF16, inputs.BF16, 0.25, base_seed=63), 1),
    (inputs.Workload("win_tc_wide", 1, 2, 2, 128, (300, 640), inputs.BF16, inputs.BF16, 0.25, base_seed=64), 5000),
    (inputs.Workload("win_tc_noncausal", 1, 2, 2, 128, (333, 520), inputs.BF16, inputs.BF16, 0.25, base_seed=65, causal=False), 130),
    (inputs.Workload("win_simt_fp32", 1, 4, 4, 64, (400, 90), inputs.FP32, inputs.FP32, 0.25, base_seed=66), 48),
]


@pytest.mark.parametrize("w,window", CASES, ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_windowed_scores_match_oracle(B, w, window):
    import torch
    dev = _dev()
    lis, q, k, _, _ = TL.stack_layers(w, range(w.n_layers), with_cache=False)
    prob = B.Problem(w.n_layers, w.n_q_heads, w.n_kv_heads, w.head_dim, w.seqlens, causal=w.causal, device=dev,
                     query_window=window)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    T = w.total_tokens
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    impls = [B.SCORE_SIMT] if w.qk_dtype == inputs.FP32 else [B.SCORE_TENSOR, B.SCORE_SIMT]
    cu = w.cu_seqlens
    for impl in impls:
        scores = torch.full((w.n_layers, w.n_q_heads, T), -1.0, dtype=torch.float32, device=dev)
        lse = torch.full_like(scores, 7.0)
        B.kvcrush_score(prob, dq, dk, scores, lse_out=lse, impl=impl, workspace=ws, status=status)
        norm = torch.empty_like(scores)
        B.kvcrush_score(prob, dq, dk, norm, normalize=True, impl=impl, workspace=ws, status=status)
        torch.cuda.synchronize()
        assert status.cpu().tolist()[0] == 0
        g, gl, gn = scores.cpu().numpy(), lse.cpu().numpy(), norm.cpu().numpy()
        for l, li in enumerate(lis):
            for s, L in enumerate(w.seqlens):
                a, b = int(cu[s]), int(cu[s + 1])
                j0 = max(0, L - window)
                c, ol = O.scores(inputs.widen(li.q[a:b], w.qk_dtype), inputs.widen(li.k[a:b], w.qk_dtype), w.causal,
                                 rows=(j0, L))
                ok = TL.within_score_tolerance(g[l][:, a:b], c)
                assert ok.all(), (w.name, impl, l, s, np.argwhere(~ok)[:4])
                np.testing.assert_allclose(gl[l][:, a + j0:b], ol[:, j0:], rtol=0, atol=3e-4)
                np.testing.assert_allclose(gn[l][:, a:b] * (L - j0), g[l][:, a:b], rtol=1e-5, atol=1e-7)
                np.testing.assert_allclose(g[l][:, a:b].astype(np.float64).sum(axis=1), float(L - j0), rtol=2e-4)


@pytest.mark.parametrize("layers,Hq,Hkv,D,seqlens,window,causal,gain", [
    (10, 16, 16, 64, (300,), 64, True, 1.0),              # one CTA alone (more units than SMs)
    (1, 4, 4, 128, (128, 129, 1000, 0, 5, 64), 64, True, 1.0),   # several sequences of very different length per cluster
    (2, 4, 1, 128, (4100,), 32, True, 1.0),               # clusters of 8, last tile of 4 keys
    (1, 2, 2, 64, (8192,), 33, True, 1.0),                # every accumulator in use
    (1, 8, 2, 128, (900, 31), 16, False, 1.0),            # 16 columns, no mask
    (6, 32, 8, 128, (1500,), 7, True, 1.0),               # units in turn on the same accumulators
    (1, 4, 2, 128, (300, 2500, 0, 5000, 90, 1100), 64, True, 1.0),       # one launch for lengths that need clusters of 1 to 8
    (6, 16, 2, 128, (300, 2500, 0, 5000, 90, 1100), 64, True, 1.0),      # a launch for each cluster size
    (20, 6, 3, 64, (1025, 1024, 2049, 31), 40, False, 1.0),              # the same at the edges between the sizes
    (1, 4, 4, 128, (700, 200), 48, True, 40.0),           # logits far outside [-100, 100]: kept tiles, exact maxima
    (1, 2, 2, 64, (600,), 64, False, 12.0),               # some tiles kept, some not
])
def test_one_pass_window_scores_match_oracle(B, layers, Hq, Hkv, D, seqlens, window, causal, gain):
    """Windows of up to 64 queries: scores within the score tolerance of the oracle, row log-sum-exp within 3e-4 (scaled by
    the gain on the queries, as the logits are)."""
    import torch
    dev = _dev()
    w = inputs.Workload("win1", layers, Hq, Hkv, D, seqlens, inputs.BF16, inputs.BF16, 0.25, base_seed=290 + D, causal=causal)
    lis, q, k, _, _ = TL.stack_layers(w, range(layers), with_cache=False)
    dq = (TL.torch_storage(q, w.qk_dtype, dev).float() * gain).to(torch.bfloat16)
    dk = TL.torch_storage(k, w.qk_dtype, dev)
    hq = dq.cpu().view(torch.int16).numpy().view(np.uint16)
    prob = B.Problem(layers, Hq, Hkv, D, seqlens, causal=causal, device=dev, query_window=window)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    scores = torch.full((layers, Hq, w.total_tokens), -1.0, dtype=torch.float32, device=dev)
    lse = torch.full_like(scores, 7.0)
    for _ in range(2):
        B.kvcrush_score(prob, dq, dk, scores, lse_out=lse, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    g, gl, cu, G = scores.cpu().numpy(), lse.cpu().numpy(), w.cu_seqlens, Hq // Hkv
    for l in sorted({0, layers - 1}):
        for s, L in enumerate(seqlens):
            a, b = int(cu[s]), int(cu[s + 1])
            if L == 0:
                continue
            j0 = max(0, L - window)
            c, ol = O.scores(inputs.widen(hq[l, a:b], w.qk_dtype), inputs.widen(lis[l].k[a:b], w.qk_dtype), causal, rows=(j0, L))
            assert TL.within_score_tolerance(g[l][:, a:b], c).all(), (l, s)
            np.testing.assert_allclose(gl[l][:, a + j0:b], ol[:, j0:], rtol=0, atol=3e-4 * gain)
            assert (gl[l][:, a:a + j0] == 7.0).all()


@pytest.mark.parametrize("layers,Hq,Hkv,D,seqlens,window,gain", [
    (12, 32, 4, 64, (700,), 64, 1.0),                     # a CTA alone, two or three units of 6 tiles through 8 accumulators
    (12, 16, 16, 64, (2000, 0, 90), 32, 1.0),             # clusters of 1 whose units differ, 16 accumulators
    (9, 32, 32, 64, (1100,), 16, 60.0),                   # logits kept in every unit, 9 tiles through 32 accumulators
    (2, 40, 8, 128, (7000,), 64, 30.0),                   # clusters of 8, 7 tiles or 6 a CTA
])
def test_units_that_follow_each_other_through_the_accumulators(B, layers, Hq, Hkv, D, seqlens, window, gain):
    """More units than clusters: the exponentials of a unit run beside the sums of the one before, accumulators are taken round
    and round, all warps share the last unit.  The CUDA-core kernels on the same inputs agree within the score tolerance."""
    import torch
    dev = _dev()
    g = torch.Generator(device=dev).manual_seed(5)
    T = sum(seqlens)
    q = (torch.randn((layers, T, Hq, D), generator=g, device=dev) * gain).to(torch.bfloat16)
    k = torch.randn((layers, T, Hkv, D), generator=g, device=dev).to(torch.bfloat16)
    prob = B.Problem(layers, Hq, Hkv, D, seqlens, device=dev, query_window=window)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    got = []
    for impl in (B.SCORE_TENSOR, B.SCORE_TENSOR, B.SCORE_SIMT):
        scores = torch.full((layers, Hq, T), -1.0, dtype=torch.float32, device=dev)
        B.kvcrush_score(prob, q, k, scores, impl=impl, workspace=ws, status=status)
        got.append(scores)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    assert torch.equal(got[0], got[1])
    assert TL.within_score_tolerance(got[0].cpu().numpy(), got[2].cpu().numpy()).all()


def test_a_few_logits_out_of_range_cost_what_their_sums_cost(B):
    """Four keys of every head whose logits of 75 are kept beside the stored exponentials (a head's attention sinks): their sums
    are formed one column after the other, the other keys go on as they are.  2.9 times the time of logits in range; value by
    value in the whole unit with a branch for each it was 6.3 times."""
    import torch
    dev = _dev()
    layers, H, L, D = 4, 32, 8192, 128
    g = torch.Generator(device=dev).manual_seed(6)
    q, k = (torch.randn((layers, L, H, D), generator=g, device=dev).to(torch.bfloat16) for _ in range(2))
    q[..., 0], k[..., 0] = 8.0, 0.0
    prob = B.Problem(layers, H, H, D, (L,), device=dev, query_window=64)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    scores = torch.empty((layers, H, L), dtype=torch.float32, device=dev)
    times = []
    for sink in (0.0, 75.0):
        k[:, :4, :, 0] = sink * D ** 0.5 / 8.0
        best = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                B.kvcrush_score(prob, q, k, scores, impl=B.SCORE_TENSOR, workspace=ws, status=status)
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b))
        times.append(min(best))
    assert status.tolist()[0] == 0
    assert times[1] < 4.5 * times[0]


@pytest.mark.parametrize("layers,seqlens,window,want", [
    (4, (8192,), 64, (1, 1)), (4, (8192,) + (300,) * 15, 64, (2, 1)), (1, (4200, 4000), 64, (1, 1)),
    (4, (8193,), 64, (2, 0)), (4, (8192,), 65, (2, 0)), (4, (8192,), 0, (2, 0)),
])
def test_score_kernel_count_follows_the_dispatch(B, layers, seqlens, window, want):
    import ctypes
    prob = B.Problem(layers, 32, 32, 128, seqlens, device=_dev(), query_window=window)
    one_pass = ctypes.c_int(-1)
    assert (B.lib().kvcrush_diag_score_kernels(prob.ref, ctypes.byref(one_pass)), one_pass.value) == want


@pytest.mark.parametrize("L,window", [
    (100, 16),                                            # one CTA alone
    (1000, 64),                                           # a cluster of 8, one tile of keys each
    (1100, 64),                                           # a cluster of 8, three CTAs without keys: their sums are on the way
])
def test_one_pass_window_waits_that_run_out_are_reported(B, L, window):
    """The bounded waits of the one-pass window kernel, made to run out through the library's diagnostic entry point: no CTA
    issues a copy, so every CTA's consumers give up, the clusters meet, tensor memory is freed and the kernel (id 4: the
    dispatch took this one) returns with the status word set and the outputs untouched.  Afterwards the public entry point
    gives the oracle's scores on the same context."""
    import ctypes
    import torch
    dev = _dev()
    fn = B.lib().kvcrush_diag_score
    vp, i32 = ctypes.c_void_p, ctypes.c_int
    fn.restype = i32
    fn.argtypes = [ctypes.POINTER(B.ProblemStruct), ctypes.POINTER(B.TensorStruct), ctypes.POINTER(B.TensorStruct),
                   vp, vp, vp, i32, i32, vp, ctypes.c_size_t, vp, vp, i32, i32]
    w = inputs.Workload("win_out", 1, 1, 1, 128, (L,), inputs.BF16, inputs.BF16, 0.25, base_seed=56)
    lis, q, k, _, _ = TL.stack_layers(w, range(1), with_cache=False)
    prob = B.Problem(1, 1, 1, 128, w.seqlens, device=dev, query_window=window)
    dq, dk = TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev)
    qs, ks = B.tensor_struct(dq), B.tensor_struct(dk)
    scores = torch.full((1, 1, L), -5.0, dtype=torch.float32, device=dev)
    lse = torch.full_like(scores, -7.0)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    stream = int(torch.cuda.current_stream().cuda_stream)
    rc = fn(prob.ref, ctypes.byref(qs), ctypes.byref(ks), None, scores.data_ptr(), lse.data_ptr(), 0, B.SCORE_TENSOR,
            ws.data_ptr(), ws.numel(), status.data_ptr(), stream, 1, 1)
    assert rc == B.OK
    torch.cuda.synchronize()
    st = status.cpu().tolist()
    assert st[0] == B.DEV_TIMEOUT and st[1] == 4 and 0 <= st[2] < 8, st
    assert bool((scores == -5.0).all()) and bool((lse == -7.0).all())
    status.zero_()
    B.kvcrush_score(prob, dq, dk, scores, lse_out=lse, workspace=ws, status=status)
    torch.cuda.synchronize()
    assert status.cpu().tolist()[0] == 0
    c, _ = O.scores(inputs.widen(lis[0].q, w.qk_dtype), inputs.widen(lis[0].k, w.qk_dtype), True, rows=(L - window, L))
    assert TL.within_score_tolerance(scores.cpu().numpy()[0], c).all()


@pytest.mark.parametrize("kernel", [1, 3, 7, 33])
def test_pooling_is_bit_exact(B, kernel):
    import torch
    dev = _dev()
    seqlens, Hq, n_layers = [300, 1, 17, 1025], 12, 2
    T = sum(seqlens)
    cu = np.concatenate([[0], np.cumsum(seqlens)])
    scores = np.zeros((n_layers, Hq, T), dtype=np.float32)
    for l in range(n_layers):
        for s, L in enumerate(seqlens):
            scores[l, :, cu[s]:cu[s + 1]] = inputs.random_scores(Hq, L, 70 + 5 * l + s)
    prob = B.Problem(n_layers, Hq, Hq, 16, seqlens, device=dev)
    out = torch.full((n_layers, Hq, T), -3.0, dtype=torch.float32, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_pool_scores(prob, torch.from_numpy(scores).to(dev), kernel, out, status=status)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for l in range(n_layers):
        for s in range(len(seqlens)):
            np.testing.assert_array_equal(got[l][:, cu[s]:cu[s + 1]], O.max_pool(scores[l][:, cu[s]:cu[s + 1]], kernel))

@pytest.mark.parametrize("seqlens,kernel", [
    ([4096], 1), ([4096], 5), ([8192], 7), ([1020], 9), ([4], 7), ([2044, 4], 33),       # quads; the last chunk in two sequences
    ([1024, 2048], 7), ([2045, 3], 7), ([1, 1023, 4096], 2047),                          # sequences that end inside a quad
    ([4096] * 80, 7), ([4095, 3, 5000] * 34, 5),                                         # chunks of 1024 tokens
    ([5000], 12001), ([4999, 2], 12001), ([3], 3),                                       # window too wide for shared memory; odd rows
])
def test_pooling_at_the_edges_of_its_chunks(B, seqlens, kernel):
    import torch
    dev = _dev()
    Hq, T = 4, sum(seqlens)
    scores = np.concatenate([inputs.random_scores(Hq, L, 90 + s) for s, L in enumerate(seqlens)], axis=1)
    prob = B.Problem(1, Hq, Hq, 16, seqlens, device=dev)
    out = torch.full((1, Hq, T), -3.0, dtype=torch.float32, device=dev)
    status = torch.zeros(4, dtype=torch.int32, device=dev)
    B.kvcrush_pool_scores(prob, torch.from_numpy(scores[None]).to(dev), kernel, out, status=status)
    torch.cuda.synchronize()
    a = 0
    for L in seqlens:
        np.testing.assert_array_equal(out[0, :, a:a + L].cpu().numpy(), O.max_pool(np.ascontiguousarray(scores[:, a:a + L]), kernel))
        a += L



@pytest.mark.parametrize("keep_recent,budgets", [(16, [(40, 30), (20, 10)]), (64, [(10, 5), (64, 64)]), (1, [(1, 1), (0, 9)])])
def test_keep_recent_selection_is_bit_exact(B, keep_recent, budgets):
    import torch
    dev = _dev()
    seqlens, Hq, Hkv = [500, 333], 32, 8
    T = sum(seqlens)
    cu = np.concatenate([[0], np.cumsum(seqlens)])
    scores = np.zeros((1, Hq, T), dtype=np.float32)
    for s, L in enumerate(seqlens):
        scores[0, :, cu[s]:cu[s + 1]] = inputs.random_scores(Hq, L, 90 + s, tie_levels=3 * s)
    b_imp = np.asarray([b[0] for b in budgets], dtype=np.int32)
    b_rep = np.asarray([b[1] for b in budgets], dtype=np.int32)
    prob = B.Problem(1, Hq, Hkv, 16, seqlens, device=dev)
    cp = B.CompressionPass(prob, b_imp[None], b_rep[None], keep_recent=keep_recent)
    ds = torch.from_numpy(scores).to(dev)
    cp.signature(ds)
    cp.select(ds)
    torch.cuda.synchronize()
    cp.check_status()
    for s, L in enumerate(seqlens):
        s32 = np.ascontiguousarray(scores[0][:, cu[s]:cu[s + 1]])
        sig = O.signatures(s32, O.thresholds(s32, int(b_imp[s] + b_rep[s])))
        idx, kind = O.select(s32, sig, int(b_imp[s]), int(b_rep[s]), Hkv, keep_recent=keep_recent)
        np.testing.assert_array_equal(cp.kept(0, s), idx.astype(np.int32))
        lo, hi = int(cp.cu_kept_host[s]), int(cp.cu_kept_host[s + 1])
        np.testing.assert_array_equal(cp.kind[lo:hi].cpu().numpy(), kind)


def test_snapkv_style_pass_end_to_end(B):
    """Window scores -> pooling -> signature -> selection with the window kept -> compaction."""
    import torch
    dev = _dev()
    w = inputs.Workload("snap", 2, 8, 2, 128, (900, 400), inputs.BF16, inputs.FP16, 0.25, base_seed=67)
    window, kernel = 32, 7
    lis, q, k, kc, vc = TL.stack_layers(w, range(2))
    prob = B.Problem(2, 8, 2, 128, w.seqlens, device=dev, query_window=window)
    b_imp, b_rep = w.budgets()
    cp = B.CompressionPass(prob, b_imp[None], b_rep[None], cache_dtype=torch.float16, pool_kernel=kernel, keep_recent=window)
    cp.run(TL.torch_storage(q, w.qk_dtype, dev), TL.torch_storage(k, w.qk_dtype, dev),
           TL.torch_storage(kc, w.cache_dtype, dev), TL.torch_storage(vc, w.cache_dtype, dev))
    torch.cuda.synchronize()
    cp.check_status()
    g = cp.scores.cpu().numpy()
    gp = cp.pooled.cpu().numpy()
    cu = w.cu_seqlens
    for l, li in enumerate(lis):
        for s, L in enumerate(w.seqlens):
            a, b = int(cu[s]), int(cu[s + 1])
            c, _ = O.scores(inputs.widen(li.q[a:b], w.qk_dtype), inputs.widen(li.k[a:b], w.qk_dtype), True,
                            rows=(L - window, L))
            assert TL.within_score_tolerance(g[l][:, a:b], c).all()
            pooled = O.max_pool(np.ascontiguousarray(g[l][:, a:b]), kernel)
            np.testing.assert_array_equal(gp[l][:, a:b], pooled)
            sig = O.signatures(pooled, O.thresholds(pooled, int(b_imp[s] + b_rep[s])))
            idx, kind = O.select(pooled, sig, int(b_imp[s]), int(b_rep[s]), 2, keep_recent=window)
            np.testing.assert_array_equal(cp.kept(l, s), idx.astype(np.int32))
            assert set(range(L - window, L)) <= set(idx[kind == 0].tolist())
            seg = l * w.n_seqs + s
            lo = int(cp.cu_kept_host[seg]) - int(cp.cu_kept_host[l * w.n_seqs])
            got = cp.k_out[l, lo:lo + len(idx)].cpu().numpy()
            assert got.tobytes() == O.compact(li.k_cache[a:b], idx).tobytes()

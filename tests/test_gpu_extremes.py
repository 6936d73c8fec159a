"""Scores of inputs that are not finite or lie at the ends of the float range: a NaN logit makes its query's log-sum-exp
NaN and with it every score the query adds to, a logit of -inf gets the weight 0, a query that does not vote has no
influence, and weights keep the relative precision of float32 down to the smallest normal number."""
import numpy as np
import pytest

from oracle import kvcrush_oracle as O
import kvc_testlib as TL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2503_00022_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def _normal(shape, seed, dtype):
    import torch
    g = np.random.Generator(np.random.Philox(seed))
    return torch.from_numpy(g.standard_normal(shape).astype(np.float32)).to("cuda:0").to(dtype)


def _score(B, q, k, lens, impl, window=0, causal=True, scale=0.0):
    """(scores, row log-sum-exp; 7.0 where a row is not written) as numpy [layers, Hq, T]."""
    import torch
    layers, T, Hq, D = q.shape
    prob = B.Problem(layers, Hq, k.shape[2], D, lens, causal=causal, softmax_scale=scale, device=q.device, query_window=window)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device=q.device)
    status = torch.zeros(4, dtype=torch.int32, device=q.device)
    scores = torch.full((layers, Hq, T), -1.0, dtype=torch.float32, device=q.device)
    lse = torch.full_like(scores, 7.0)
    B.kvcrush_score(prob, q, k, scores, lse_out=lse, impl=impl, workspace=ws, status=status)
    assert status.cpu().tolist()[0] == 0
    return scores.cpu().numpy(), lse.cpu().numpy()


def _decode(B, q_new, k, scale=0.0):
    import torch
    layers, L, _, D = k.shape
    prob = B.Problem(layers, q_new.shape[2], k.shape[2], D, (L,), softmax_scale=scale, device=k.device)
    scores = torch.zeros((layers, q_new.shape[2], L), dtype=torch.float32, device=k.device)
    status = torch.zeros(4, dtype=torch.int32, device=k.device)
    B.kvcrush_score_decode(prob, q_new, k, scores, status=status)
    return scores.cpu().numpy()


# The column of a NaN key is chosen so that its exponential takes the special-function unit: the polynomial that serves
# columns 6, 7, 14 and 15 of every 16 clamps its argument and with it a NaN.
@pytest.mark.parametrize("layers,Hq,L,p", [
    (1, 2, 201, 64), (1, 2, 201, 160),       # blocks of one tile: four slots a quarter
    (1, 8, 1100, 128), (1, 32, 2052, 513),   # blocks of one or two tiles
    (8, 32, 2052, 1024),                     # full blocks, the last one with a single tile
])
def test_nan_key_reaches_every_row_that_sees_it_on_the_tensor_cores(B, layers, Hq, L, p):
    import torch
    q, k = _normal((layers, L, Hq, 128), 1, torch.bfloat16), _normal((layers, L, Hq, 128), 2, torch.bfloat16)
    k[:, p] = float("nan")
    s, lse = _score(B, q, k, (L,), B.SCORE_TENSOR)
    assert np.isfinite(lse[..., :p]).all() and np.isnan(lse[..., p:]).all()
    assert np.isnan(s).all()


@pytest.mark.parametrize("layers,Hq,L,p,causal", [
    (1, 1, 600, 70, True), (1, 1, 600, 3, False),     # streamed tiles shared by a cluster
    (4, 40, 130, 0, True), (4, 40, 130, 127, True),   # one block per tile of rows; a row whose every logit is NaN
])
def test_nan_key_reaches_every_row_that_sees_it_on_the_cuda_cores(B, layers, Hq, L, p, causal):
    import torch
    q, k = _normal((layers, L, Hq, 64), 3, torch.float32), _normal((layers, L, Hq, 64), 4, torch.float32)
    k[:, p] = float("nan")
    s, lse = _score(B, q, k, (L,), B.SCORE_SIMT, causal=causal)
    first = p if causal else 0
    assert np.isfinite(lse[..., :first]).all() and np.isnan(lse[..., first:]).all()
    assert np.isnan(s).all()


def test_queries_that_do_not_vote_have_no_influence_on_the_cuda_cores(B):
    """The window starts inside a tile of 64 queries; one of the tile's other queries is NaN, one gives infinite logits."""
    import torch
    L, window = 200, 50
    q, k = _normal((1, L, 2, 64), 5, torch.float32), _normal((1, L, 2, 64), 6, torch.float32)
    want, want_lse = _score(B, q, k, (L,), B.SCORE_SIMT, window=window)
    q[:, 130] = float("nan")
    q[:, 140] = 3e38
    got, got_lse = _score(B, q, k, (L,), B.SCORE_SIMT, window=window)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(got_lse, want_lse)


@pytest.mark.parametrize("lens,window,causal", [
    ((200, 150), 0, True), ((200, 150), 0, False), ((1001, 130, 77), 0, True),     # the next sequence's queries in the last tile
    ((1001, 600), 100, True), ((300, 400), 260, True),                             # and queries before the window in the first one
    ((256, 150), 0, True), ((384, 77), 128, True),                                 # full tiles: none of either kind
])
@pytest.mark.parametrize("layers,Hq", [(1, 2), (16, 32)])                          # blocks of one or two tiles, full blocks
@pytest.mark.parametrize("bad", [float("nan"), 3e38])
def test_queries_that_do_not_vote_have_no_influence_on_the_tensor_cores(B, lens, window, causal, layers, Hq, bad):
    """Tiles of the column sweep hold the next sequence's first queries and queries before the window; here those give NaN or
    infinite logits.  The row sweep may take another reference for the rows beside them, and the polynomial that serves a
    quarter of its exponentials is off by 7.5e-5 to either side, by the fraction of its argument."""
    import torch
    T = sum(lens)
    q, k = _normal((layers, T, Hq, 64), 23, torch.bfloat16), _normal((layers, T, Hq, 64), 24, torch.bfloat16)
    want, want_lse = _score(B, q, k, lens, B.SCORE_TENSOR, window=window, causal=causal)
    first = lens[0]
    at = [first + i for i in range(0, 40, 3)]                # in both exponentials' columns
    if window:
        at += [first - window - 1 - i for i in range(0, 40, 3)]
    q[:, at] = bad
    got, got_lse = _score(B, q, k, lens, B.SCORE_TENSOR, window=window, causal=causal)
    np.testing.assert_allclose(got_lse[..., :first], want_lse[..., :first], rtol=0, atol=1.5e-4)
    np.testing.assert_allclose(got[..., :first], want[..., :first], rtol=2e-4)


@pytest.mark.parametrize("L,window,p", [(100, 16, 50), (1000, 64, 0), (4000, 33, 3333), (300, 64, 290)])
def test_nan_key_reaches_every_voting_row_of_a_window(B, L, window, p):
    import torch
    q, k = _normal((2, L, 4, 128), 7, torch.bfloat16), _normal((2, L, 4, 128), 8, torch.bfloat16)
    k[:, p] = float("nan")
    s, lse = _score(B, q, k, (L,), B.SCORE_TENSOR, window=window)
    first = max(L - window, p)                                  # first voting row that sees the key
    assert np.isfinite(lse[..., L - window:first]).all() and np.isnan(lse[..., first:]).all()
    assert (lse[..., :L - window] == 7.0).all()
    assert np.isnan(s).all()


@pytest.mark.parametrize("what", ["nan", "inf"])
def test_a_query_without_finite_sum_touches_the_keys_it_sees_only(B, what):
    """A NaN query, and one with a single logit of +inf (no other of its logits is out of range).  Blocks that see the NaN
    recompute their weights instead of reading stored ones, a quarter of which come from a polynomial of 7.5e-5."""
    import torch
    L, window, j = 300, 64, 270
    q, k = _normal((1, L, 2, 64), 9, torch.bfloat16), _normal((1, L, 2, 64), 10, torch.bfloat16)
    q[..., 0], k[..., 0] = 0.0, 0.0
    want, _ = _score(B, q, k, (L,), B.SCORE_TENSOR, window=window)
    if what == "nan":
        q[:, j] = float("nan")
    else:
        q[:, j, :, 0], k[:, 17, :, 0] = 1e30, 1e30
    s, lse = _score(B, q, k, (L,), B.SCORE_TENSOR, window=window)
    assert np.isnan(lse[..., j]).all() and np.isfinite(np.delete(lse, j, axis=-1)).all()
    assert np.isnan(s[..., :j + 1]).all()
    np.testing.assert_allclose(s[..., j + 1:], want[..., j + 1:], rtol=1e-4)


@pytest.mark.parametrize("lens,window", [
    ((300, 200), 40), ((300, 200), 20), ((300, 200), 5),     # the window ends inside its 64, 32 or 16 columns
    ((50, 300, 37), 64), ((1100, 900), 40),                  # a sequence shorter than the window; a cluster of CTAs
])
@pytest.mark.parametrize("bad", [float("nan"), 3e38])
def test_queries_of_the_next_sequence_have_no_influence_on_a_window(B, lens, window, bad):
    """The columns behind a window's last query hold the next sequence's first queries; here those give NaN or infinite
    logits.  Blocks that hold such logits recompute the others' weights instead of reading stored ones, a quarter of which
    come from a polynomial of 7.5e-5: in the sums over keys and over queries."""
    import torch
    T = sum(lens)
    q, k = _normal((1, T, 2, 64), 21, torch.bfloat16), _normal((1, T, 2, 64), 22, torch.bfloat16)
    want, want_lse = _score(B, q, k, lens, B.SCORE_TENSOR, window=window)
    ends = np.cumsum(lens)
    for e in ends[:-1]:
        q[:, e] = bad                                        # votes in its own sequence only where that is as short as the window
        q[:, e + 2] = -bad
    got, got_lse = _score(B, q, k, lens, B.SCORE_TENSOR, window=window)
    first = ends[0]
    np.testing.assert_allclose(got_lse[..., :first], want_lse[..., :first], rtol=0, atol=1e-4)
    np.testing.assert_allclose(got[..., :first], want[..., :first], rtol=2e-4)
    if len(lens) == 2:                                       # those queries do not vote: the second sequence is as before
        np.testing.assert_allclose(got[..., first:], want[..., first:], rtol=2e-4)


@pytest.mark.parametrize("window,shallow", [(16, 0), (40, 0), (16, 8), (40, 20)])
def test_small_weights_of_a_window_keep_their_value_beside_a_huge_logit(B, window, shallow):
    """32 keys with logits of 110 (2^158) fill one block; the others' logits of 60 to 63 stay in the range that is stored as
    2^x.  Their weights of e^-50 have to come out as such: exponentials of 7.5e-5, logits rounded by 2^-24 of 158.  The first
    `shallow` of the voting queries see half of every logit."""
    import torch
    L = 512
    q, k = torch.zeros((1, L, 1, 64), device="cuda:0"), torch.zeros((1, L, 1, 64), device="cuda:0")
    q[..., 0] = 1.0
    q[:, L - window:L - window + shallow, :, 0] = 0.5
    k[0, :, 0, 0] = 60.0 + 0.25 * (torch.arange(L, device="cuda:0") % 13)
    k[0, 64:96, 0, 0] = 110.0
    q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
    s, _ = _score(B, q, k, (L,), B.SCORE_TENSOR, window=window, scale=1.0)
    want, _ = O.scores(q[0].double().cpu().numpy(), k[0].double().cpu().numpy(), True, scale=1.0, rows=(L - window, L))
    np.testing.assert_allclose(s[0, 0], want[0], rtol=3e-4)


@pytest.mark.parametrize("dtype,L,Hq", [("float32", 2048, 2), ("bfloat16", 2048, 2), ("bfloat16", 52000, 8)])
def test_decode_keys_with_logits_of_minus_infinity_get_no_weight(B, dtype, L, Hq):
    """A stretch of keys longer than one block's part, and (52000 keys x 8 heads) the variant without stored logits."""
    import torch
    q, k = _normal((1, 1, Hq, 64), 11, torch.float32), _normal((1, L, 1, 64), 12, torch.float32)
    q[..., 0], k[..., 0] = 1e30, 0.0
    n = L // 8 * 3
    k[:, n:2 * n, :, 0] = -1e30                                  # product -1e60: -inf in float32
    q, k = q.to(getattr(torch, dtype)), k.to(getattr(torch, dtype))
    got = _decode(B, q, k)[0]
    assert (got[:, n:2 * n] == 0.0).all()
    rest = torch.cat([k[0, :n], k[0, 2 * n:]]).double().cpu().numpy()
    want = O.decode_update(np.zeros((Hq, L - n)), q[0, 0].double().cpu().numpy(), rest)
    np.testing.assert_allclose(np.delete(got, np.s_[n:2 * n], axis=1), want, rtol=1e-4)


@pytest.mark.parametrize("L,Hq,first,last", [(2048, 2, 5, 6), (2048, 2, 256, 512), (52000, 8, 5, 6), (52000, 8, 6512, 13024)])
def test_decode_nan_keys_reach_every_score_of_the_sequence(B, L, Hq, first, last):
    """A single key, and all the keys of the second of a cluster's eight blocks."""
    import torch
    q, k = _normal((1, 1, Hq, 64), 13, torch.bfloat16), _normal((1, L, 1, 64), 14, torch.bfloat16)
    k[:, first:last] = float("nan")
    assert np.isnan(_decode(B, q, k)).all()


def test_decode_adds_weights_below_the_smallest_normal_number(B):
    """Logits of 0 (one key) and -88 to -100: weights down to e^-100 = 2^-144.  Their last place is 2^-149: two of it from the
    exponential, half of it each from the factor of the block and from the product.  A second step adds the same again."""
    import torch
    L = 400
    q, k = torch.zeros((1, 1, 1, 8), device="cuda:0"), torch.zeros((1, L, 1, 8), device="cuda:0")
    q[..., 0] = 1.0
    k[0, 1:, 0, 0] = -88.0 - 12.0 * torch.arange(1, L, device="cuda:0") / L
    prob = B.Problem(1, 1, 1, 8, (L,), softmax_scale=1.0, device="cuda:0")
    scores = torch.zeros((1, 1, L), dtype=torch.float32, device="cuda:0")
    status = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    w = np.exp(k[0, :, 0, 0].double().cpu().numpy())
    w /= w.sum()
    for n in (1, 2):
        B.kvcrush_score_decode(prob, q, k, scores, status=status)
        got = scores.cpu().numpy()[0, 0].astype(np.float64)
        assert (np.abs(got - n * w) <= 1e-5 * n * w + 3 * n * 2.0 ** -149).all()


def test_one_long_and_many_short_sequences_on_the_cuda_cores(B):
    """512 tiles of rows x 4096 sequences x 4096 heads would be more blocks than a grid holds; the work is small (a window of
    one query).  Layers and heads share their rows, so every slice gives the same scores."""
    import torch
    layers, Hq, long_len, n_short = 32, 128, 32768, 4095
    T = long_len + n_short
    q = _normal((1, T, 1, 8), 15, torch.float32).expand(layers, T, Hq, 8)
    k = _normal((1, T, 1, 8), 16, torch.float32).expand(layers, T, Hq, 8)
    lens = (long_len,) + (1,) * n_short
    prob = B.Problem(layers, Hq, Hq, 8, lens, device="cuda:0", query_window=1)
    ws = torch.empty(B.kvcrush_workspace_size(prob, B.STAGE_SCORE), dtype=torch.uint8, device="cuda:0")
    status = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    scores = torch.full((layers, Hq, T), -1.0, dtype=torch.float32, device="cuda:0")
    B.kvcrush_score(prob, q, k, scores, impl=B.SCORE_SIMT, workspace=ws, status=status)
    assert bool((scores == scores[:1, :1]).all())
    got = scores[0, 0].cpu().numpy()
    want, _ = O.scores(q[0, :long_len, :1].double().cpu().numpy(), k[0, :long_len, :1].double().cpu().numpy(), True,
                       rows=(long_len - 1, long_len))
    assert TL.within_score_tolerance(got[:long_len], want[0]).all()
    np.testing.assert_allclose(got[long_len:], 1.0, rtol=1e-6)

"""Sizes at which the kernels' splits change, against the float64 oracle.

Rows on and off the 16-byte grid, launches around one and two rows per SM (the
row kernel's CTA sizes), draws over a whole row by clusters of every size, the
float32 rows that the general kernel takes by depth histogram, payloads and
nuclei around the ranking limits, branch caches whose threshold comes from a
sample, and the sparse resample on ragged rows.  Everything is compared under
the rules of tests/parity.py (ids, lengths, tokens and branches bit for bit).
"""
import numpy as np
import pytest

import gen
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FALLBACK, RADIX, LAZY, SCANNED, DEPTH, DEPTH_LOST = 0, 4, 5, 13, 14, 15   # words of the workspace's path counters


@pytest.fixture(scope="module")
def A():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_02514_gb300 as A
    A.load()
    return A


def _dev(x, offset=0):
    """x on the GPU, its first element `offset` elements past an aligned address."""
    t = torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) if x.dtype == np.uint16 else torch.from_numpy(x).cuda()
    if offset == 0:
        return t
    big = torch.empty(t.numel() + offset, dtype=t.dtype, device="cuda")
    big[offset:].copy_(t.reshape(-1))
    return big[offset:].view(t.shape)


def _verify(A, orc, w, inp, offset=0, q_offset=0):
    z, q = _dev(inp["z"], offset), _dev(inp["q"], q_offset)
    xt, u = _dev(inp["xt"]), _dev(inp["u"])
    ws = torch.zeros(A.workspace_bytes(w.B, w.K, w.V, w.k), dtype=torch.uint8, device="cuda")
    g = A.verify(z, q, xt, u, w.T, w.top_p, w.k, workspace=ws)
    torch.cuda.synchronize()
    g = {key: v.cpu().numpy() for key, v in g.items()}
    o = orc.verify(inp["z"], inp["q"], inp["xt"], inp["u"], w.T, w.top_p, w.k)
    res = parity.compare_verify(inp, g, o, w.top_p, inp["z"].dtype == np.uint16, w.k)
    counters = ws[A.COUNTERS_OFFSET:A.COUNTERS_OFFSET + 64].view(torch.int32).cpu().numpy().tolist()
    return res, counters, o


def _logits(z, dtype):
    z = np.ascontiguousarray(z, dtype=np.float32)
    return gen.f32_to_bf16(z) if dtype == "bf16" else z


# ---------------------------------------------------------------------------
# rows off the 16-byte grid


@pytest.mark.parametrize("dtype,V,offset", [
    ("bf16", 5, 1), ("bf16", 2047, 0), ("bf16", 2049, 3), ("bf16", 65537, 7), ("bf16", 65544, 4),
    ("f32", 3, 1), ("f32", 8191, 0), ("f32", 8195, 2), ("f32", 32769, 3), ("f32", 32772, 1)])
@pytest.mark.parametrize("top_p", [0.9, 1.0])
def test_rows_off_the_grid(A, orc, dtype, V, offset, top_p):
    # K = 8: the rows start at every offset from a 16-byte boundary
    w = gen.make_workload(3, 8, V, dtype, T=0.8, top_p=top_p, k=min(V, 24), seed=81)
    inp = gen.generate(w)
    res, counters, _ = _verify(A, orc, w, inp, offset, q_offset=offset % 4)
    # (rows of a few ids may have no positive logit: the general kernel's)
    assert res["checked_seqs"] >= 1 and (V < 100 or counters[FALLBACK] == 0), (res, counters)


# ---------------------------------------------------------------------------
# the row kernel's CTA sizes


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("per_sm,extra", [(1, 0), (1, 1), (2, 0), (2, 2)])
def test_launches_around_whole_rows_per_sm(A, orc, dtype, per_sm, extra):
    n = torch.cuda.get_device_properties(0).multi_processor_count
    B = (per_sm * n + 2 * extra) // 2        # K = 1: two rows a sequence
    w = gen.make_workload(B, 1, 9000, dtype, T=0.8, top_p=0.9, k=20, seed=82)
    res, _, _ = _verify(A, orc, w, gen.generate(w))
    assert res["checked_seqs"] >= 0.8 * B


# ---------------------------------------------------------------------------
# draws over a whole row


@pytest.mark.parametrize("B", [1, 39, 80, 170])       # clusters of 8, 4, 2, and more sequences than clusters
@pytest.mark.parametrize("dtype,V,top_p", [("bf16", 16384, 0.9), ("bf16", 16387, 1.0), ("f32", 8200, 0.9)])
def test_draws_over_a_whole_row(A, orc, B, dtype, V, top_p):
    w = gen.make_workload(B, 1, V, dtype, T=1.6, top_p=top_p, k=8, seed=83)
    inp = gen.generate(w)
    res, counters, o = _verify(A, orc, w, inp)
    n = o["n_nuc"][np.arange(B), o["accept_len"]]
    assert (n > 512).all() and counters[SCANNED] + counters[FALLBACK] >= B, counters
    # (an id at the crossing carries about 2e-5 of the mass, so a row's two
    # cumulative sums lie within 1e-6 of top_p in about 1 row of 10: 2 x 2e-6 /
    # 2e-5 / 2; a sequence has up to two such rows)
    assert res["checked_seqs"] >= 0.7 * B, res


def test_draw_without_residual_and_with_a_bad_draft_row(A, orc):
    # q = 1 everywhere: the residual is zero and the token comes from p; then
    # a NaN and a negative q inside row 0's nucleus, and one outside it
    w = gen.make_workload(6, 1, 16384, "bf16", T=1.6, top_p=0.9, k=8, seed=84)
    inp = gen.generate(w)
    q = inp["q"].copy()
    q[:3] = 1.0
    zf = gen.bf16_to_f32(inp["z"])
    order = [np.lexsort((np.arange(w.V), -zf[b, 0].astype(np.float64))) for b in range(w.B)]
    for b in (3, 4, 5):                       # rejected at row 0: its draft token is the least likely id
        inp["xt"][b, 0] = order[b][-1]
        q[b, 0, order[b][-1]] = 0.5
    q[3, 0, order[3][100]] = np.nan
    q[4, 0, order[4][200]] = -0.25
    q[5, 0, order[5][-2]] = -0.25
    inp["q"] = q
    z, qt, xt, u = _dev(inp["z"]), _dev(q), _dev(inp["xt"]), _dev(inp["u"])
    g = A.verify(z, qt, xt, u, w.T, w.top_p, w.k)
    o = orc.verify(inp["z"], q, inp["xt"], inp["u"], w.T, w.top_p, w.k)
    assert (o["accept_len"][3:] == 0).all()
    for key in ("accept_len", "out_token", "row_status"):
        np.testing.assert_array_equal(g[key].cpu().numpy(), o[key], err_msg=key)
    assert (o["out_token"][[3, 4]] == -1).all() and o["out_token"][5] >= 0


# ---------------------------------------------------------------------------
# float32 rows handed to the general kernel


@pytest.mark.parametrize("V,offset,shift,top_p", [
    (40000, 0, 0.0, 0.97), (40003, 1, 0.0, 0.97), (40000, 0, -300.0, 0.97), (40000, 0, 4000.0, 0.6), (40000, 0, 0.0, 1.0)])
def test_float32_rows_by_depth_histogram(A, orc, V, offset, shift, top_p):
    # flat rows (T = 2): nuclei of thousands of ids, more than the row kernel
    # lists; logits far from zero on either side
    w = gen.make_workload(4, 2, V, "f32", T=2.0, top_p=top_p, k=40, seed=85)
    inp = gen.generate(w)
    inp["z"] = (inp["z"] + np.float32(shift)).astype(np.float32)
    res, counters, o = _verify(A, orc, w, inp, offset)
    if top_p < 1.0:
        assert counters[FALLBACK] == 12 and (o["n_nuc"] > 4096).any(), counters
    assert counters[DEPTH] == counters[FALLBACK] and res["checked_seqs"] >= 2, (res, counters)


def test_bfloat16_rows_by_depth_histogram(A, orc):
    # normal logits at T = 1: the crossing lies among negative ones, out of the
    # value histogram's reach, and no value is shared by many ids
    w = gen.make_workload(3, 2, 20000, "bf16", T=1.0, top_p=0.9, k=40, seed=92, sigma=1.0)
    res, counters, _ = _verify(A, orc, w, gen.generate(w))
    assert counters[FALLBACK] == 9 and counters[DEPTH] == 9 and res["checked_seqs"] >= 1, (res, counters)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_rows_of_alike_values_are_declined_before_the_second_read(A, orc, dtype):
    # 8 values: thousands of ids of each, more than either list holds; the binned
    # path (2048 ids a bin) does not hold them either
    w = gen.make_workload(4, 2, 40000, dtype, T=1.0, top_p=0.8, k=40, seed=93)
    inp = gen.generate(w)
    z = np.random.default_rng(93).integers(0, 8, inp["z"].shape).astype(np.float32) * 0.25 + 1.0
    inp["z"] = _logits(z, dtype)
    res, counters, _ = _verify(A, orc, w, inp)
    assert counters[FALLBACK] == 12 and counters[RADIX] == 12, counters
    assert counters[DEPTH] == 0 and counters[DEPTH_LOST] == 0 and res["checked_seqs"] >= 1, (res, counters)


@pytest.mark.parametrize("B", [20, 100, 250])          # CTAs of 1024, 512 and 256 threads
@pytest.mark.parametrize("V", [40000, 40003])
def test_float32_rows_whose_records_overflow(A, orc, B, V):
    # equal logits everywhere: every chunk is recorded until the records are
    # full, and the warps stop recording while others still add to them.  (An
    # id carries 2.5e-5 of the mass and the crossing lies inside one, so only
    # draws within 1e-6 of an id's end, one in 12, are flagged.)
    w = gen.make_workload(B, 1, V, "f32", T=1.0, top_p=0.9001125, k=8, seed=90)
    inp = gen.generate(w)
    inp["z"] = np.full_like(inp["z"], 1.5)
    res, counters, _ = _verify(A, orc, w, inp)
    assert counters[FALLBACK] == 2 * B and res["checked_seqs"] >= 0.6 * B, (res, counters)


# ---------------------------------------------------------------------------
# the cut is the one of the row's exact mass


@pytest.mark.parametrize("dtype,V", [("f32", 20000), ("f32", 20001), ("bf16", 20001), ("bf16", 50003)])
@pytest.mark.parametrize("n", [256, 510, 2048, 12000])
@pytest.mark.parametrize("exact", [False, True])
def test_cut_at_half_of_equal_masses(A, dtype, V, n, exact):
    # n ids of one value each, top_p = 1/2: exactly n / 2 of them are the
    # nucleus.  A total wrong in its last bits moves the cut to n / 2 + 1 in
    # half the rows (half a last bit of float32 is 6e-8, an id's share 1e-4)
    B, k = 80, 64
    rng = np.random.default_rng(n)
    z = np.full((B, 2, V), -np.inf, np.float32)
    for b in range(B):
        for i in range(2):
            ids = rng.choice(V, n, replace=False) if b % 2 else rng.integers(V - n + 1) + np.arange(n)
            z[b, i, ids] = rng.uniform(0.3, 9.0)
    zt = _dev(_logits(z, dtype))
    q = torch.full((B, 1, V), 1.0 / V, device="cuda")
    xt, u = torch.zeros(B, 1, dtype=torch.int32, device="cuda"), torch.full((B, 2), 0.5, device="cuda")
    g = A.verify(zt, q, xt, u, 0.7, 0.5, k, exact=exact)
    p = g["topk_probs"].cpu().numpy().astype(np.float64)
    assert (np.abs(p * (n // 2) - 1.0) < 1e-6).all(), np.unique(np.round(1.0 / p, 2))


@pytest.mark.parametrize("dtype,V,sigma,T,top_p", [
    ("f32", 40000, 3.0, 0.9, 0.9), ("f32", 40003, 3.0, 0.9, 0.9),
    ("f32", 40000, 1.0, 1.0, 0.8), ("bf16", 40003, 3.0, 0.9, 0.9), ("bf16", 40003, 3.0, 0.9, 1.0), ("bf16", 40003, 1.0, 1.0, 0.8)])
@pytest.mark.parametrize("B", [40, 300])               # one wave, and rows that see finished ones
def test_a_row_is_the_same_whichever_kernel_finishes_it(A, dtype, V, sigma, T, top_p, B):
    # repeated calls (the rows that overflow the row kernel's areas depend on
    # what has finished before) and the general kernel alone: the same bits.
    # (Not float32 rows with top_p = 1: their last bit may depend on the kernel.)
    w = gen.make_workload(B, 2, V, dtype, T=T, top_p=top_p, k=24, seed=91, sigma=sigma, rho=0.9)
    inp = gen.generate(w)
    z, q, xt, u = (_dev(inp[key]) for key in ("z", "q", "xt", "u"))
    first = None
    for run in range(5):
        g = A.verify(z, q, xt, u, w.T, w.top_p, w.k, exact=run == 4)
        if first is None:
            first = g
        for key in first:
            assert torch.equal(g[key], first[key]), (key, run)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B", [20, 50, 250])           # CTAs of 1024, 512 and 256 threads
@pytest.mark.parametrize("top_p", [0.9, 1.0])
def test_rows_whose_sample_is_masked(A, orc, dtype, B, top_p):
    # the row kernel's sample is tiles 3 t mod 128, t < 64, of 32 chunks: all of
    # it -inf, a few ids left outside it; every third row keeps all its ids, so
    # that the depths of finished rows are known
    V = 128 * 32 * (8 if dtype == "bf16" else 4)
    w = gen.make_workload(B, 4, V, dtype, T=0.9, top_p=top_p, k=16, seed=89)
    inp = gen.generate(w)
    rng = np.random.default_rng(89)
    z = (rng.standard_normal((B, 5, V)) * 3.0).astype(np.float32)
    tile = np.arange(V) // (V // 128)
    out = np.flatnonzero(~np.isin(tile, 3 * np.arange(64) % 128))
    for r in range(B * 5):
        if r % 3:
            row = z[r // 5, r % 5]
            keep = rng.choice(out, 40, replace=False)
            left = row[keep].copy()
            row[:] = -np.inf
            row[keep] = left
    inp["z"] = _logits(z, dtype)
    res, _, _ = _verify(A, orc, w, inp)
    assert res["checked_seqs"] >= 0.9 * B


# ---------------------------------------------------------------------------
# payloads and nuclei around the ranking limits


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n", [1, 3, 128, 509, 512, 513, 1023, 1025])
def test_nuclei_around_the_ranking_limits(A, orc, dtype, n):
    # n ids hold nearly all the mass, at a few values (ties go by id)
    V = 20000
    w = gen.make_workload(3, 1, V, dtype, T=1.0, top_p=0.9999, k=256, seed=86)
    inp = gen.generate(w)
    rng = np.random.default_rng(86)
    z = np.full((3, 2, V), -60.0, np.float32)
    for b in range(3):
        for i in range(2):
            z[b, i, rng.choice(V, n, replace=False)] = 4.0 + 0.03125 * rng.integers(0, 40, n)
    inp["z"] = _logits(z, dtype)
    res, _, o = _verify(A, orc, w, inp)
    assert res["checked_seqs"] == 3 and (np.abs(o["n_nuc"] - n) <= 0.001 * n + 1).all()


@pytest.mark.parametrize("V,k", [(5, 5), (64, 64), (256, 256), (2048, 256), (4100, 200), (102400, 1), (600000, 256)])
def test_payload_of_top_p_one_rows(A, orc, V, k):
    # k = V (the payload is the row), fewer groups than k, one chunk a group, ragged, and groups of
    # several iterations
    w = gen.make_workload(2, 1, V, "bf16", T=1.0, top_p=1.0, k=k, seed=87)
    res, _, _ = _verify(A, orc, w, gen.generate(w))
    assert res["checked_seqs"] == 2


# ---------------------------------------------------------------------------
# branch caches


def _cache(A, orc, q, xt, F, offset=0):
    c = A.cache_build(_dev(q, offset), _dev(xt), F)
    torch.cuda.synchronize()
    obt, obp = orc.cache_build(q, xt, F)
    parity.compare_cache(c["branch_tok"].cpu().numpy(), c["branch_prob"].cpu().numpy(), obt, obp)


@pytest.mark.parametrize("V,offset", [(2, 0), (33, 1), (8191, 0), (8192, 0), (8197, 3), (65537, 0), (70000, 2)])
@pytest.mark.parametrize("B", [1, 10, 320])            # clusters of 8, 4 and one CTA a row
def test_cache_rows_around_the_sample(A, orc, V, offset, B):
    rng = np.random.default_rng(V + B)
    K = 2
    q = rng.random((B, K, V)).astype(np.float32) ** 8
    q[0, 0, rng.random(V) < 0.9] = 0.0                 # few positive ids
    q[-1, 1, :] = 0.0                                  # one
    q[-1, 1, V // 2] = 0.25
    q /= np.maximum(q.sum(-1, keepdims=True), 1e-30) * 1.0001
    xt = rng.integers(0, V, size=(B, K)).astype(np.int32)
    _cache(A, orc, q.astype(np.float32), xt, [min(5, V - 1), min(70, V - 1)], offset)


@pytest.mark.parametrize("B", [1, 320])
def test_cache_rows_that_mislead_the_sample(A, orc, B):
    # equal values everywhere (more than the candidates' room), a sample far
    # above and one far below the rest of the row, a NaN and a negative value
    V, K = 40000, 4
    rng = np.random.default_rng(88)
    q = rng.random((B, K, V)).astype(np.float32) * 1e-6
    q[:, 0] = 1.0 / V
    q[:, 1, :256 * 4] += 1e-3                          # the first sampled block holds the largest
    q[:, 2, 256 * 4:512 * 4] += 1e-4                   # a block outside the sample does
    q[:, 3, 17] = -1.0
    xt = np.full((B, K), 5, np.int32)
    _cache(A, orc, q, xt, [9, 64, 64, 64])


# ---------------------------------------------------------------------------
# sparse resample


@pytest.mark.parametrize("V,offset", [(7, 1), (1001, 0), (4099, 3), (33000, 0), (33003, 2)])
def test_resample_on_ragged_rows(A, orc, V, offset):
    # payloads that end before the nucleus does (the tail is spread), with the
    # first and the last id of the row among them
    B, K, k = 12, 2, min(6, V)
    rng = np.random.default_rng(V)
    q = rng.random((B, K, V)).astype(np.float32) ** 4
    q /= q.sum(-1, keepdims=True)
    ids = np.stack([rng.permutation(np.concatenate([[0, V - 1], 1 + rng.choice(V - 2, k - 2, replace=False)]))
                    for _ in range(B * (K + 1))]).reshape(B, K + 1, k).astype(np.int32)
    probs = np.sort(rng.random((B, K + 1, k)), axis=-1)[..., ::-1].astype(np.float32)
    probs = (probs / probs.sum(-1, keepdims=True) * 0.6).astype(np.float32)
    tail = np.full((B, K + 1), 0.4, np.float32)
    tail[0] = 0.0
    al = rng.integers(0, K + 1, B).astype(np.int32)
    st = np.zeros((B, K + 1), np.int32)
    u = (rng.integers(1, 1 << 24, (B, K + 1)) / float(1 << 24)).astype(np.float32)
    o = orc.resample_sparse(al, ids, probs, tail, st, q, u)
    g = A.resample_sparse(_dev(al), _dev(ids), _dev(probs), _dev(tail), _dev(st), _dev(q, offset), _dev(u))
    np.testing.assert_array_equal(g["status"].cpu().numpy(), o["status"])
    tok = g["token"].cpu().numpy()
    near = np.array([any(np.isfinite(c) and abs(o["res_target"][b] - c) < 1e-6 * o["res_sum"][b]
                         for c in (o["res_cj"][b], o["res_cjm1"][b])) for b in range(B)])
    assert (tok == o["token"])[~near].all() and near.sum() <= 2


@pytest.mark.parametrize("V", [1001, 152064])
def test_resample_with_a_bad_draft_value_outside_the_payload(A, orc, V):
    # a NaN or a negative value that one thread of one CTA meets, at the start,
    # in the middle and at the end of the row: the whole cluster gives the row up
    bad = [0, 5, 31, 32, V // 3, V // 2, V - 2, V - 1]
    B, K, k = 2 * len(bad) + 1, 1, 4
    rng = np.random.default_rng(V + 1)
    q = rng.random((B, K, V)).astype(np.float32)
    q /= q.sum(-1, keepdims=True)
    for i, x in enumerate(bad):
        q[2 * i, 0, x] = np.nan
        q[2 * i + 1, 0, x] = -1e-3
    ids = np.tile(np.array([100, 200, 300, 400], np.int32), (B, K + 1, 1))
    probs = np.full((B, K + 1, k), 0.15, np.float32)
    tail = np.full((B, K + 1), 0.4, np.float32)
    al, st = np.zeros(B, np.int32), np.zeros((B, K + 1), np.int32)
    u = np.full((B, K + 1), 0.25, np.float32)
    o = orc.resample_sparse(al, ids, probs, tail, st, q, u)
    g = A.resample_sparse(_dev(al), _dev(ids), _dev(probs), _dev(tail), _dev(st), _dev(q), _dev(u))
    np.testing.assert_array_equal(g["status"].cpu().numpy(), o["status"])
    assert (g["status"].cpu().numpy()[:-1] != 0).all() and g["status"][-1] == 0
    assert (g["token"].cpu().numpy()[:-1] == -1).all()

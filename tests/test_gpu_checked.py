"""The checked build on small and ragged cases.

libacespec_checked.so is the library compiled with -DACES_CHECKED: every
data-dependent shared- and global-memory index of every kernel (row kernels,
draws, cache, resample, KV compaction) is checked against its array's
bound, and the first index out of range is recorded (site, index, bound)
instead of used.  Nothing traps.  These tests build it (about a minute),
route the package's calls to it, run the small and ragged parity cases, the
path cases and the other entry points, compare with the float64 oracle, and
require the record to stay empty.  The build also counts the rows of q that
the branch cache reads again, which the last tests here look at.
"""
import dataclasses

import numpy as np
import pytest

import gen
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def A():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_02514_gb300 as A
    from paper_2609_02514_gb300 import build
    build.build(checked=True)
    A.use_checked(True)
    A.checked_violation()  # start from an empty record
    yield A
    A.use_checked(False)


def _dev(inp):
    z = inp["z"]
    zt = torch.from_numpy(z.view(np.int16)).cuda().view(torch.bfloat16) if z.dtype == np.uint16 \
        else torch.from_numpy(z).cuda()
    return zt, torch.from_numpy(inp["q"]).cuda(), torch.from_numpy(inp["xt"]).cuda(), torch.from_numpy(inp["u"]).cuda()


def _verify_all(A, orc, w, inp, exact=False):
    z, q, xt, u = _dev(inp)
    g = A.verify(z, q, xt, u, w.T, w.top_p, w.k, exact=exact)
    F = tuple(min(3, w.V - 1) for _ in range(w.K))
    c = A.cache_build(q, xt, F)
    slot = A.cache_lookup(c["branch_tok"], F, g["accept_len"], g["out_token"])
    rs = A.resample_sparse(g["accept_len"], g["topk_ids"], g["topk_probs"], g["tail_mass"], g["row_status"], q, u)
    torch.cuda.synchronize()
    assert A.checked_violation() is None
    gn = {key: v.cpu().numpy() for key, v in g.items()}
    o = orc.verify(inp["z"], inp["q"], inp["xt"], inp["u"], w.T, w.top_p, w.k)
    parity.compare_verify(inp, gn, o, w.top_p, inp["z"].dtype == np.uint16, w.k)
    obt, obp = orc.cache_build(inp["q"], inp["xt"], F)
    parity.compare_cache(c["branch_tok"].cpu().numpy(), c["branch_prob"].cpu().numpy(), obt, obp)
    np.testing.assert_array_equal(slot.cpu().numpy(),
                                  orc.cache_lookup(c["branch_tok"].cpu().numpy(), F, gn["accept_len"], gn["out_token"]))
    assert rs["token"].shape == (w.B,)


CASES = [
    dict(B=1, K=4, V=32000, dtype="f32", T=1.0, top_p=1.0, k=16),       # the first workload's shape
    dict(B=3, K=2, V=10007, dtype="f32", T=0.7, top_p=0.9, k=37),       # unaligned rows: general path
    dict(B=2, K=3, V=4099, dtype="bf16", T=1.3, top_p=0.95, k=5),       # unaligned bf16 rows
    dict(B=4, K=5, V=8200, dtype="bf16", T=0.6, top_p=0.8, k=64),       # aligned, ragged last tile
    dict(B=2, K=16, V=20000, dtype="f32", T=1.0, top_p=1.0, k=256),     # top_p = 1, largest payload
    dict(B=5, K=1, V=65544, dtype="bf16", T=2.0, top_p=0.99, k=16),     # flat rows: exact fallback
    dict(B=3, K=4, V=128256, dtype="bf16", T=1.0, top_p=0.9, k=32, sigma=3.0, rho=0.5),  # value mode
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: f"{c['dtype']}_V{c['V']}_p{c['top_p']}")
def test_no_index_out_of_range(A, orc, cfg):
    cfg = dict(cfg)
    w = gen.make_workload(cfg.pop("B"), cfg.pop("K"), cfg.pop("V"), seed=13, **cfg)
    inp = gen.generate(w)
    _verify_all(A, orc, w, inp)
    _verify_all(A, orc, w, inp, exact=True)


def test_no_index_out_of_range_on_degenerate_rows(A, orc):
    w = gen.make_workload(8, 3, 4096, "f32", T=1.0, top_p=0.9, k=8, seed=21)
    inp = dict(gen.generate(w))
    z, q, xt, u = (inp[key].copy() for key in ("z", "q", "xt", "u"))
    z[0, 1, 17] = np.nan
    z[1, 0, :] = -np.inf
    z[2, 2, 5] = np.inf
    z[3, 0, ::2] = -np.inf
    xt[4, 0] = 4096 + 3
    q[5, 0, xt[5, 0]] = 0.0
    z[7, :, :] = 0.5
    inp.update(z=z, q=q, xt=xt, u=u)
    zt, qt, xtt, ut = _dev(inp)
    A.verify(zt, qt, xtt, ut, w.T, w.top_p, w.k)
    torch.cuda.synchronize()
    assert A.checked_violation() is None


def test_no_index_out_of_range_in_the_edge_kernels(A):
    # KV compaction and the tree mask on a small tree (hits, misses, full accept)
    B, K, H, D, planes, t0 = 4, 3, 2, 64, 2, 8
    F = [2, 2, 1]
    bl = K + 1
    S = t0 + K + sum(F) * bl
    kv = torch.randn(planes, B, H, S, D, device="cuda").to(torch.bfloat16)
    pref = torch.full((B,), t0, dtype=torch.int32, device="cuda")
    al = torch.tensor([0, 1, 3, 2], dtype=torch.int32, device="cuda")
    slot = torch.tensor([1, -1, -2, 4], dtype=torch.int32, device="cuda")
    A.compact_kv(kv, pref, al, slot, K, bl)
    A.tree_mask(F, bl)
    torch.cuda.synchronize()
    assert A.checked_violation() is None


# ---------------------------------------------------------------------------
# branch caches: rows that are read again


def _cache(A, orc, q, F, seed=0):
    """Branches against the oracle; returns the number of rows read again."""
    B, K, V = q.shape
    xt = np.random.default_rng(seed).integers(0, V, size=(B, K)).astype(np.int32)
    A.checked_cache_selects()
    c = A.cache_build(torch.from_numpy(q).cuda(), torch.from_numpy(xt).cuda(), F)
    torch.cuda.synchronize()
    n = A.checked_cache_selects()
    assert A.checked_violation() is None
    obt, obp = orc.cache_build(q, xt, F)
    parity.compare_cache(c["branch_tok"].cpu().numpy(), c["branch_prob"].cpu().numpy(), obt, obp)
    return n


def _rows(kind, B, K, V, seed):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        q = rng.random((B, K, V), dtype=np.float32)
    elif kind == "equal":
        q = np.ones((B, K, V), np.float32)
    else:
        z = rng.standard_normal((B, K, V), dtype=np.float32) * (1.0 if kind == "likely ids first" else 3.0)
        if kind == "likely ids first":
            z -= 1.1 * np.log(np.arange(1, V + 1, dtype=np.float32))
        if kind == "likely ids in the sample":  # half a block of it, when a row has one CTA
            z[:, :, 512:1024] += 15.0
        q = np.exp(z - z.max(-1, keepdims=True))
    return (q / q.sum(-1, keepdims=True) * np.float32(0.999)).astype(np.float32)


@pytest.mark.parametrize("V", [4100, 8000, 8192, 16384])
@pytest.mark.parametrize("F", [256, 512, 1024])
@pytest.mark.parametrize("B", [1, 50, 100, 200])       # clusters of 8 (as V allows), 4, 2 and one CTA a row
def test_wide_fanouts_of_short_rows_are_read_once(A, orc, V, F, B):
    # the sample is the whole slice, and up to four of the values asked for share
    # each of the 256 maxima: how many do varies, most on the shortest rows
    n = _cache(A, orc, _rows("normal", B, 2, V, V + F + B), [F, F])
    assert n <= {256: 0, 512: B // 25, 1024: B // 2}[F], n


@pytest.mark.parametrize("kind,B,V,F,again", [
    ("uniform", 1, 256000, 8, False), ("uniform", 20, 256000, 8, False), ("uniform", 170, 40000, 200, False),
    ("equal", 1, 40000, 4, False), ("equal", 170, 40000, 64, False), ("equal", 170, 30001, 300, False),
    ("equal", 5, 1 << 20, 1024, True), ("likely ids first", 170, 33001, 64, False),
    ("likely ids first", 1, 128256, 512, True), ("likely ids in the sample", 170, 33001, 400, True)])
def test_rows_of_alike_values_and_rows_the_sample_misleads(A, orc, kind, B, V, F, again):
    n = _cache(A, orc, _rows(kind, B, 2, V, V + F), [F, 0])
    assert n == (B if again else 0), n


def test_rows_read_again_to_every_digit(A, orc):
    # the first eighth of a row holds the largest values, so the eight CTAs'
    # thresholds are too high; they span 2^23, 2^19, 2^8 and one bit patterns, so
    # that one, two, three and four digits (the last: of the id) are counted.
    # Then a row with fewer positive values than branches, and one with a
    # negative value and thousands of NaN
    B, V, F = 6, 60000, 700
    rng = np.random.default_rng(5)
    q = np.zeros((B, 1, V), np.float32)
    for b, lim in enumerate([1 << 23, 1 << 19, 1 << 8, 1]):
        bits = np.uint32(0x3A800000) + rng.integers(0, lim, V).astype(np.uint32)
        bits[:7000] += np.uint32(lim)
        q[b, 0] = bits.view(np.float32)
    q[4, 0, rng.choice(V, 300, replace=False)] = rng.random(300).astype(np.float32) * 1e-3
    q[5, 0] = _rows("likely ids first", 1, 1, V, 6)[0, 0]
    q[5, 0, 7] = -0.5
    assert _cache(A, orc, q, [F]) == 5
    nan = np.concatenate([[100], np.arange(1000, V, 3)])
    q[5, 0, nan] = np.nan
    c = A.cache_build(torch.from_numpy(q).cuda(), torch.full((B, 1), 3, dtype=torch.int32, device="cuda"), [F])
    torch.cuda.synchronize()
    assert A.checked_violation() is None
    tok = c["branch_tok"].cpu().numpy()
    assert not np.isin(tok[5], nan).any() and (tok[5] >= 0).all() and (tok[4] >= 0).sum() == 300

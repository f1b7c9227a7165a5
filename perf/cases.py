"""Timed cases of the AceSpec path: what a user of this package calls, over the range it is called with.

A case names the call (`op`) and its sizes:

  verify    verify(): the cloud checks the drafted chains of B requests and packs the downlink payload
  step      cloud_step() and cache_lookup(): verification with the branch cache of the same batch
  sparsify  sparsify(): the payload alone, for B rows of logits
  draft     cache_build() and tree_mask(): the edge prepares its branches before the reply arrives
  edge      resample_sparse(), cache_lookup() and compact_kv(): the edge takes the reply in

Logits and draft distributions follow the recipe of gen/workloads.py (correlated normal logits, an
optional Zipf head, a draft distribution with or without a support cut), made on the GPU.
"""
import math

import torch

import paper_2609_02514_gb300 as A

MAX_ELEMS = 256 * 17 * 256000      # logits (or draft probabilities) of the largest case
MAX_RAGGED = MAX_ELEMS // 16       # of a drawn case whose rows are not 16-byte multiples
DEV = "cuda"


def _verify(name, B, K, V, dtype, T, top_p, k, sigma=3.0, rho=0.8, zipf=False, cut=1e-4, op="verify", F0=4, decay=1.0):
    return dict(name=name, op=op, B=B, K=K, V=V, dtype=dtype, T=T, top_p=top_p, k=k, sigma=sigma, rho=rho,
                zipf=zipf, cut=cut, F0=F0, decay=decay)


def listed():
    return [
        # one interactive request, plain sampling: latency of the whole cloud side
        _verify("step_b1_k4_v32000_f32", 1, 4, 32000, "f32", 1.0, 1.0, 16, rho=0.95, op="step", F0=2),
        # a small server with float32 logits
        _verify("verify_b16_k8_v32000_f32", 16, 8, 32000, "f32", 0.8, 0.9, 32),
        # a mid-sized batch with peaked rows (Zipf head): one partial wave of rows
        _verify("verify_b64_k8_v152064", 64, 8, 152064, "bf16", 0.7, 0.95, 64, sigma=4.0, rho=0.7, zipf=True),
        # flat rows and many rejections: nuclei of thousands of ids
        _verify("verify_b128_k16_v128256", 128, 16, 128256, "bf16", 1.0, 0.9, 32, rho=0.5),
        # plain sampling (top_p = 1): the nucleus is the whole vocabulary
        _verify("verify_b32_k4_v102400_p1", 32, 4, 102400, "bf16", 1.0, 1.0, 64, rho=0.9),
        # a vocabulary whose rows are not 16-byte multiples
        _verify("verify_b24_k5_v50003", 24, 5, 50003, "bf16", 0.8, 0.9, 32),
        # large-batch verification: the cloud alone
        _verify("verify_b256_k16_v256000", 256, 16, 256000, "bf16", 0.6, 0.8, 128, rho=0.9),
        # the whole cloud step at full load
        _verify("step_b256_k16_v256000", 256, 16, 256000, "bf16", 0.6, 0.8, 128, rho=0.9, op="step"),
        # payload of float32 rows (a logits service without drafts)
        dict(name="sparsify_r256_v128256_f32", op="sparsify", B=256, V=128256, dtype="f32", T=0.7, top_p=0.95, k=64,
             sigma=3.0, rho=0.9, zipf=False),
        # an edge device drafting for one user
        dict(name="draft_b1_k16_v128256", op="draft", B=1, K=16, V=128256, F0=6, decay=0.95, T=1.0, sigma=3.0,
             zipf=False, cut=1e-4),
        # a drafting server with wide fan-outs and a draft sampler of full support
        dict(name="draft_b64_k8_v152064_f64", op="draft", B=64, K=8, V=152064, F0=64, decay=1.0, T=0.7, sigma=4.0,
             zipf=True, cut=0.0),
        # the edge side of a reply: draw from the payload, look the branch up, move its KV rows
        dict(name="edge_b32_k8_v152064", op="edge", B=32, K=8, V=152064, F0=4, decay=1.0, T=0.7, top_p=0.95, k=32,
             sigma=4.0, rho=0.9, zipf=True, cut=1e-4, planes=16, H=8, D=128, prefix=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["verify"] * 5 + ["step"] * 2 + ["sparsify"] * 2 + ["draft"] * 3 + ["edge"] * 2)
    dtype = rng.choice(["bf16", "bf16", "f32"])
    V = _log(rng, 8000, 262144)
    if rng.random() < 0.65:
        V -= V % 64
    K = rng.randint(1, 16)
    rows = 1 if op == "sparsify" else K + 1
    esz = 2 if dtype == "bf16" else 4
    most = MAX_ELEMS // (2 if dtype == "f32" and op != "draft" else 1)
    if (V * esz) % 16 != 0:
        most = MAX_RAGGED
    if op in ("step", "draft", "edge") and V % 4 != 0:
        most = MAX_RAGGED
    if op == "edge":
        most = min(most, 64 * rows * V)
    B = _log(rng, 1, max(1, min(4096 if op == "sparsify" else 256, most // (rows * V))))
    c = dict(op=op, B=B, V=V, T=round(rng.uniform(0.5, 1.2), 3), sigma=round(rng.uniform(2.5, 4.0), 3),
             zipf=rng.random() < 0.3)
    if op != "sparsify":
        c["K"] = K
        c["cut"] = rng.choice([1e-4, 1e-4, 0.0])
    if op != "draft":
        c["top_p"] = rng.choice([0.8, 0.9, 0.95, 1.0, round(rng.uniform(0.6, 0.99), 4)])
        c["k"] = _log(rng, 8, 256)
        c["rho"] = round(rng.uniform(0.5, 0.97), 3)
    if op in ("verify", "step", "sparsify"):
        c["dtype"] = dtype
    if op in ("step", "draft", "edge"):
        c["F0"] = _log(rng, 1, 8 if op != "draft" or rng.random() < 0.5 else 128)
        c["decay"] = rng.choice([1.0, 0.95, 0.8])
    while "F0" in c and sum(_fanout(c)) * (K + 1) > 6000:
        c["F0"] //= 2
    if op == "edge":
        c.update(planes=rng.choice([8, 16]), H=rng.choice([2, 8]), D=rng.choice([64, 128]),
                 prefix=rng.choice([128, 512]))
        c["B"] = min(B, max(1, 40000 // _kv_positions(c)))
    return c


def _kv_positions(case):
    return case["prefix"] + case["K"] + sum(_fanout(case)) * (case["K"] + 1)


def _fanout(case):
    return tuple(max(1, int(round(case["F0"] * case["decay"] ** d))) for d in range(case["K"]))


def _logits(case, n, rows, g):
    """Draft and target logits [n, rows, V], float32."""
    V, sigma = case["V"], case["sigma"]
    zd = torch.randn(n, rows, V, generator=g, device=DEV)
    zd *= sigma
    z = None
    if "rho" in case:
        z = torch.randn(n, rows, V, generator=g, device=DEV)
        z *= math.sqrt(1.0 - case["rho"] ** 2) * sigma
        z.add_(zd, alpha=case["rho"])
    return zd, z


def _zipf(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed * 7 + 3)
    ids = torch.randperm(case["V"], generator=g, device=DEV)[:100]
    rank = torch.arange(1, ids.numel() + 1, device=DEV, dtype=torch.float32)
    return ids, 2.0 * torch.log((ids.numel() + 1.0) / rank)


def _inputs(case, seed):
    """z [B, K+1, V] (absent for draft), q [B, K, V], xt [B, K], u [B, K+1]."""
    op, B, V = case["op"], case["B"], case["V"]
    K = case.get("K", 0)
    rows = K if op == "draft" else K + 1
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)
    dt = torch.bfloat16 if case.get("dtype") == "bf16" else torch.float32
    keep_z = op != "draft"
    z = torch.empty(B, rows, V, dtype=dt, device=DEV) if keep_z else None
    q = torch.empty(B, K, V, device=DEV) if K else None
    xt = torch.empty(B, K, dtype=torch.int32, device=DEV) if K else None
    head = _zipf(case, int(seed)) if case["zipf"] else None
    step = max(1, (1 << 27) // (rows * V))
    for b0 in range(0, B, step):
        n = min(step, B - b0)
        zd, zt = _logits(case, n, rows, g)
        if head is not None:
            zd[:, :, head[0]] += head[1]
            if zt is not None:
                zt[:, :, head[0]] += head[1]
        if keep_z:
            z[b0:b0 + n] = zt
        if K:
            w = zd[:, :K]
            w = torch.exp((w - w.amax(-1, keepdim=True)) / case["T"])
            if case["cut"] > 0.0:
                w[w < case["cut"]] = 0.0
            w /= w.sum(-1, keepdim=True)
            q[b0:b0 + n] = w
            xt[b0:b0 + n] = torch.multinomial(w.view(-1, V), 1, generator=g).view(n, K).to(torch.int32)
    u = torch.randint(1, 1 << 24, (B, K + 1), generator=g, device=DEV).float() / float(1 << 24)
    return z, q, xt, u, g


def _payload(case, z, pi):
    """What verify() packs for row pi of every sequence (float32), in 64-bit arithmetic."""
    B, V, k = case["B"], case["V"], case["k"]
    ids = torch.full((B, case["K"] + 1, k), -1, dtype=torch.int32, device=DEV)
    probs = torch.zeros(B, case["K"] + 1, k, device=DEV)
    tail = torch.zeros(B, case["K"] + 1, device=DEV)
    for b in range(B):
        i = int(pi[b])
        order, p, n = _nucleus(z[b, i:i + 1], case["T"], case["top_p"])
        m = min(int(n[0]), k)
        ids[b, i, :m] = order[0, :m].to(torch.int32)
        probs[b, i, :m] = p[0, :m].float()
        tail[b, i] = 0.0 if int(n[0]) <= k else float(1.0 - p[0, :m].sum())
    return ids, probs, tail


def _branches(case, q, xt):
    """Branch tokens as cache_build() lays them out (the largest q besides the draft token)."""
    F = _fanout(case)
    cols = []
    for d, f in enumerate(F):
        row = q[:, d].clone()
        row.scatter_(1, xt[:, d:d + 1].long(), -1.0)
        v, i = row.topk(min(f, case["V"] - 1), dim=-1)
        cols.append(torch.where(v > 0, i, torch.full_like(i, -1)).to(torch.int32))
    return torch.cat(cols, dim=1).contiguous()


def prepare(case, seed):
    op, B, V = case["op"], case["B"], case["V"]
    K = case.get("K", 0)
    z, q, xt, u, g = _inputs(case, seed)
    s = dict(case=case, op=op, z=z, q=q, xt=xt, u=u)
    if op in ("step", "draft", "edge"):
        s["F"] = _fanout(case)
    if op in ("verify", "step", "sparsify"):
        if op == "sparsify":
            s["z"] = z.view(B, V)
        # a serving loop keeps its scratch
        s["ws"] = torch.zeros(A.workspace_bytes(B, K, V, case["k"]), dtype=torch.uint8, device=DEV)
    if op == "edge":
        # the reply: a geometric accepted length, that row's payload
        r = torch.rand(B, K, generator=g, device=DEV)
        pi = (r < 0.75).int().cumprod(1).sum(1).to(torch.int32)
        s["pi"] = pi
        s["ids"], s["probs"], s["tail"] = _payload(case, z, pi)
        s["status"] = torch.zeros(B, K + 1, dtype=torch.int32, device=DEV)
        s["bt"] = _branches(case, q, xt)
        L = K + 1
        s["kv"] = torch.empty(case["planes"], B, case["H"], _kv_positions(case), case["D"], device=DEV,
                              dtype=torch.bfloat16).normal_(generator=g)
        s["prefix"] = torch.randint(case["prefix"] // 2, case["prefix"] + 1, (B,), generator=g,
                                    device=DEV).to(torch.int32)
        s["L"] = L
        s["z"] = None  # the edge has no target logits
    return s


def run(s):
    c, op = s["case"], s["op"]
    if op == "verify":
        return A.verify(s["z"], s["q"], s["xt"], s["u"], c["T"], c["top_p"], c["k"], workspace=s["ws"])
    if op == "step":
        o = A.cloud_step(s["z"], s["q"], s["xt"], s["u"], c["T"], c["top_p"], c["k"], s["F"], workspace=s["ws"])
        o["slot"] = A.cache_lookup(o["branch_tok"], s["F"], o["accept_len"], o["out_token"])
        return o
    if op == "sparsify":
        return A.sparsify(s["z"], c["T"], c["top_p"], c["k"], workspace=s["ws"])
    if op == "draft":
        o = A.cache_build(s["q"], s["xt"], s["F"])
        o["mask"], o["depth"] = A.tree_mask(s["F"], c["K"] + 1)
        return o
    o = A.resample_sparse(s["pi"], s["ids"], s["probs"], s["tail"], s["status"], s["q"], s["u"])
    o["slot"] = A.cache_lookup(s["bt"], s["F"], s["pi"], o["token"])
    o["new_len"] = A.compact_kv(s["kv"], s["prefix"], s["pi"], o["slot"], c["K"], s["L"])
    o["kv"] = s["kv"]
    return o


def work(case):
    op, B, V = case["op"], case["B"], case["V"]
    K = case.get("K", 0)
    k = case.get("k", 0)
    rows = B * (K + 1)
    es = 2 if case.get("dtype") == "bf16" else 4
    S = sum(_fanout(case)) if "F0" in case and op in ("step", "draft", "edge") else 0
    cache = B * K * V * 4 + B * K * 4 + B * S * 8
    out = rows * (8 * k + 8) + B * 8
    if op in ("verify", "step"):
        by = rows * V * es + B * K * 12 + rows * 4 + out
        fl = 4 * rows * V
        if op == "step":
            by += cache + B * 4
            fl += B * K * V
        return dict(bytes=by, flops=fl)
    if op == "sparsify":
        return dict(bytes=rows * V * es + out, flops=4 * rows * V)
    if op == "draft":
        n = K + S * (K + 1)
        return dict(bytes=cache + n * ((n + 31) // 32) * 4 + n * 4, flops=B * K * V)
    # the payloads, the draft row of the (nearly all) rejecting sequences whose nucleus passes k ids,
    # and the KV rows of about a third of the sequences (the hits), read and written
    kv = 2 * case["planes"] * case["H"] * (K + 1) * case["D"] * 2
    return dict(bytes=B * (12 * k + 32) + B * V * 4 + (B // 3) * kv, flops=4 * B * V)


def tolerance(case):
    if case["op"] == "draft":
        return {"rel": 2e-7}  # one fp32 subtraction and division: 4e-8 seen
    if case["op"] == "edge":
        return "exact"  # tokens, slots and moved rows
    # fp32 exp-sums: 1e-7 seen, 7e-7 when one row's nucleus ends an id earlier or later (mass within
    # 1e-7 of top_p); such a row may change one payload id
    return {"rel": 3e-6, "differ": 1e-4}


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits


def _nucleus(z, T, top_p):
    """rows [n, V] -> ids in (logit desc, id asc) order, their probabilities in the nucleus, its size."""
    v, order = torch.sort(z.float() + 0.0, dim=-1, descending=True, stable=True)
    w = torch.exp((v.double() - v[:, :1].double()) / T)
    S = w.sum(-1, keepdim=True)
    if top_p >= 1.0:
        n = torch.isfinite(v).sum(-1)
        p = w / S
    else:
        c = torch.cumsum(w, -1)
        n = ((c < float(torch.tensor(top_p, dtype=torch.float32)) * S).sum(-1) + 1).clamp(max=z.shape[-1])
        Sn = torch.gather(c, 1, (n - 1).unsqueeze(1))
        p = torch.where(torch.arange(z.shape[-1], device=z.device).unsqueeze(0) < n.unsqueeze(1), w / Sn,
                        torch.zeros((), dtype=torch.float64, device=z.device))
    return order, p, n


def _pick(w, u):
    """Smallest id whose prefix sum exceeds u times the total."""
    c = torch.cumsum(w, 0)
    return int(torch.searchsorted(c, u * c[-1], right=True).clamp(max=w.numel() - 1))


def _exact_verify(case, z, q, xt, u):
    B, K, V, k = case["B"], case["K"], case["V"], case["k"]
    T = float(torch.tensor(case["T"], dtype=torch.float32))
    i32 = dict(dtype=torch.int32, device=DEV)
    o = dict(accept_len=torch.zeros(B, **i32), out_token=torch.zeros(B, **i32), row_status=torch.zeros(B, K + 1, **i32),
             topk_ids=torch.full((B, K + 1, k), -1, **i32),
             topk_probs=torch.zeros(B, K + 1, k, dtype=torch.float64, device=DEV),
             tail_mass=torch.zeros(B, K + 1, dtype=torch.float64, device=DEV))
    for b in range(B):
        order, p, n = _nucleus(z[b], T, case["top_p"])
        _payload64(o, b, order, p, n, k)
        ps = torch.zeros(K + 1, V, dtype=torch.float64, device=DEV).scatter_(1, order, p)
        qx = torch.gather(q[b].double(), 1, xt[b].long().unsqueeze(1)).squeeze(1)
        px = torch.gather(ps[:K], 1, xt[b].long().unsqueeze(1)).squeeze(1)
        acc = u[b, :K].double() < torch.clamp(px / qx, max=1.0)
        pi = int(acc.int().cumprod(0).sum())
        r = ps[pi]
        if pi < K:
            res = torch.clamp(ps[pi] - q[b, pi].double(), min=0.0)
            r = res if float(res.sum()) > 0.0 else r
        o["accept_len"][b] = pi
        o["out_token"][b] = _pick(r, float(u[b, K]))
    return o


def _payload64(o, b, order, p, n, k):
    m = torch.arange(k, device=DEV).unsqueeze(0) < n.unsqueeze(1)
    o["topk_ids"][b] = torch.where(m, order[:, :k], torch.full_like(order[:, :k], -1)).to(torch.int32)
    o["topk_probs"][b] = torch.where(m, p[:, :k], torch.zeros_like(p[:, :k]))
    o["tail_mass"][b] = torch.where(n <= k, torch.zeros_like(p[:, 0]), p[:, k:].sum(-1))


def _exact_cache(case, q, xt):
    bt = _branches(case, q, xt)
    F = _fanout(case)
    d = torch.repeat_interleave(torch.arange(len(F), device=DEV), torch.tensor(F, device=DEV))
    den = 1.0 - torch.gather(q, 2, xt.long().unsqueeze(2)).squeeze(2).double()
    v = q[:, d].gather(2, bt.clamp(min=0).long().unsqueeze(2)).squeeze(2).double() / den[:, d]
    return dict(branch_tok=bt, branch_prob=torch.where(bt >= 0, v, torch.zeros_like(v)))


def _exact_lookup(case, bt, pi, tok):
    F = _fanout(case)
    off = [sum(F[:d]) for d in range(len(F) + 1)]
    slot = torch.full_like(pi, -1)
    for b in range(case["B"]):
        i = int(pi[b])
        if i == case["K"]:
            slot[b] = -2
            continue
        hit = torch.nonzero(bt[b, off[i]:off[i + 1]] == tok[b])
        if hit.numel() and int(tok[b]) >= 0:
            slot[b] = off[i] + int(hit[0])
    return slot


def _exact_mask(F, L):
    K = len(F)
    start = [d for d in range(K) for _ in range(F[d])]
    n = K + len(start) * L
    m = torch.zeros(n, (n + 31) // 32 * 32, dtype=torch.bool)
    depth = torch.zeros(n, dtype=torch.int32)
    for i in range(K):
        m[i, :i + 1] = True
        depth[i] = i
    low = torch.tril(torch.ones(L, L, dtype=torch.bool))
    for s, d in enumerate(start):
        at = K + s * L
        m[at:at + L, :d] = True
        m[at:at + L, at:at + L] = low
        depth[at:at + L] = torch.arange(d, d + L, dtype=torch.int32)
    bits = (m.view(n, -1, 32).long() << torch.arange(32)).sum(-1)
    return torch.where(bits >= 1 << 31, bits - (1 << 32), bits).to(torch.int32), depth


def exact(case, seed):
    op = case["op"]
    s = prepare(case, seed)
    if op in ("verify", "step"):
        o = _exact_verify(case, s["z"], s["q"], s["xt"], s["u"])
        if op == "step":
            o.update(_exact_cache(case, s["q"], s["xt"]))
            o["slot"] = _exact_lookup(case, o["branch_tok"], o["accept_len"], o["out_token"])
        return o
    if op == "sparsify":
        B, V, k = case["B"], case["V"], case["k"]
        o = dict(topk_ids=torch.empty(B, k, dtype=torch.int32, device=DEV),
                 topk_probs=torch.empty(B, k, dtype=torch.float64, device=DEV),
                 tail_mass=torch.empty(B, dtype=torch.float64, device=DEV),
                 row_status=torch.zeros(B, dtype=torch.int32, device=DEV))
        T = float(torch.tensor(case["T"], dtype=torch.float32))
        step = max(1, (1 << 24) // V)
        for b in range(0, B, step):
            part = slice(b, min(B, b + step))
            _payload64(o, part, *_nucleus(s["z"][part], T, case["top_p"]), k)
        return o
    if op == "draft":
        o = _exact_cache(case, s["q"], s["xt"])
        m, d = _exact_mask(s["F"], case["K"] + 1)
        o["mask"], o["depth"] = m, d
        return o
    B, K, V = case["B"], case["K"], case["V"]
    tok = torch.zeros(B, dtype=torch.int32, device=DEV)
    for b in range(B):
        i = int(s["pi"][b])
        ids = s["ids"][b, i]
        m = ids >= 0
        I, P, tau = ids[m].long(), s["probs"][b, i][m].double(), float(s["tail"][b, i])
        w = torch.zeros(V, dtype=torch.float64, device=DEV)
        if i < K:
            q = s["q"][b, i].double()
            if tau > 0.0:
                out = torch.ones(V, dtype=torch.bool, device=DEV)
                out[I] = False
                rest = float(q[out].sum())
                w = q * max(0.0, tau / rest - 1.0) if rest > 0.0 else w
            w[I] = torch.clamp(P - q[I], min=0.0)
        if i == K or float(w.sum()) == 0.0:
            w.zero_()
            w[I] = P
        tok[b] = _pick(w, float(s["u"][b, K]))
    o = dict(token=tok, status=torch.zeros(B, dtype=torch.int32, device=DEV))
    o["slot"] = _exact_lookup(case, s["bt"], s["pi"], tok)
    kv, L = s["kv"], s["L"]
    new_len = torch.zeros(B, dtype=torch.int32, device=DEV)
    for b in range(B):
        t, i, sl = int(s["prefix"][b]), int(s["pi"][b]), int(o["slot"][b])
        if sl >= 0:
            src = t + K + sl * L
            kv[:, b, :, t + i:t + i + L] = kv[:, b, :, src:src + L].clone()
            new_len[b] = t + i + L
        else:
            new_len[b] = t + (K if sl == -2 else i)
    o["new_len"], o["kv"] = new_len, kv
    return o

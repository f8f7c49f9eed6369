"""Timed cases of the per-chunk 2-bit KV-cache path.

A program that uses the package runs, for each attention layer and chunk of a
video: attention of the chunk's Queries over the packed history and the active
chunk (once per denoising step), and at the chunk boundary the Query
statistics and basis, the k-means tables and the quantize-append of the
finished chunk.  The cases are these calls, each through its public entry
point, and one whole rollout of a short clip.  ``listed`` names them, ``draw``
gives others of the same ranges, ``exact`` the 64-bit results in plain torch.

Inputs follow the repository's synthetic recipe (synth.py), drawn on the GPU:
Queries N(0,1) times LogNormal(0, 0.5) channel scales, Keys N(0,1) with four
channels eight times larger (Student-t(3) there for ``tail``), Values N(0,1).
"""
import math

import torch

import paper_2609_26425_gb300 as qwm

D = 128
DEV = "cuda"


def _case(name, op, heads, tokens, past=0, queries=0, cur=0, centroids=64, group=32, rank=16, cands=4, two_level=False,
          tail=False, window=False, iters=10, lse=False):
    c = {"op": op, "heads": heads, "tokens": tokens, "past": past, "queries": queries, "cur": cur,
         "centroids": centroids, "group": group, "rank": rank, "cands": cands, "two_level": two_level, "tail": tail,
         "window": window, "iters": iters, "lse": lse}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one denoising step of the smallest configuration: 4 heads, two cached chunks and the active one
        _case("attend_h4", "attend", 4, 880, past=2, queries=880, cur=880),
        # one layer of a 1.3B causal DiT with its 15-frame sliding window full
        _case("attend_dit", "attend", 12, 880, past=15, queries=880, cur=880, rank=8, tail=True, window=True),
        # one layer of a Wan-14B shaped DiT, six cached chunks of 3 latent frames
        _case("attend_wan14b", "attend", 40, 4680, past=6, queries=4680, cur=4680, centroids=256),
        # few Queries over a long history (a late, small chunk of a long video)
        _case("attend_long", "attend", 40, 4680, past=14, queries=1024, cur=1024, centroids=256),
        # odd sizes, the two-level scale format, wide groups, the largest rank, log-sum-exp wanted, no active chunk
        _case("attend_ragged", "attend", 16, 1337, past=5, queries=1001, centroids=100, group=64, rank=32,
              two_level=True, lse=True),
        # quantize-append of one finished chunk: the smallest configuration, the Wan-14B layer, and a long chunk
        # with the other storage options and more candidates
        _case("append_h4", "append", 4, 880),
        _case("append_wan14b", "append", 40, 4680, centroids=256),
        _case("append_16k", "append", 40, 16001, centroids=64, group=64, rank=32, cands=8, two_level=True),
        # k-means tables of one chunk's Keys (the boundary fits Keys and Values)
        _case("fit_h4", "fit", 4, 880),
        _case("fit_wan14b", "fit", 40, 4680, centroids=256),
        # Query statistics of one chunk, then the weights and the principal basis
        _case("basis_wan14b", "basis", 40, 4680, centroids=256),
        # a whole short clip: three chunks of one 1.3B DiT layer, every step of the lifecycle
        _case("rollout_dit", "rollout", 12, 880, past=3, rank=8, tail=True),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["attend", "attend", "attend", "append", "append", "fit", "basis", "rollout"])
    heads = rng.choice([4, 8, 12, 16, 24, 32, 40])
    opt = {"centroids": rng.choice([16, 64, 100, 256]), "rank": rng.choice([0, 8, 16, 16, 32]),
           "group": rng.choice([32, 32, 64]), "two_level": rng.random() < 0.25, "tail": rng.random() < 0.3}
    if op == "attend":
        while True:
            tokens, past = log(300, 6000), log(1, 16)
            queries = tokens if rng.random() < 0.6 else log(100, 6000)
            cur = 0 if rng.random() < 0.2 else queries
            keys = past * tokens + cur
            if heads * queries * keys <= 40 * 4680 * 32760 and heads * past * tokens <= 40 * 65520:
                break
        return _case("", op, heads, tokens, past, queries, cur, window=rng.random() < 0.3, lse=rng.random() < 0.3, **opt)
    if op == "append":
        return _case("", op, heads, log(300, 16000), cands=rng.choice([1, 2, 4, 4, 8]), **opt)
    if op == "fit":
        return _case("", op, heads, log(300, 4680), iters=rng.choice([4, 10]), **opt)
    if op == "basis":
        return _case("", op, heads, log(300, 8000), **opt)
    return _case("", op, rng.choice([4, 8, 12]), log(300, 1600), rng.choice([2, 3, 4]), **opt)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


class _Source:
    """The seeded Queries, Keys and Values of one layer."""

    def __init__(self, case, seed):
        self.case, self.g = case, _gen(seed)
        H = case["heads"]
        self.scale = torch.exp(0.5 * torch.randn(H, D, generator=self.g, device=DEV))
        self.outliers = torch.randperm(D, generator=self.g, device=DEV)[:4]

    def randn(self, *shape):
        return torch.randn(*shape, generator=self.g, device=DEV)

    def queries(self, n):
        return (self.randn(n, self.case["heads"], D) * self.scale).bfloat16()

    def keys(self, n):
        k = self.randn(n, self.case["heads"], D)
        if self.case["tail"]:
            z = self.randn(n, self.case["heads"], 4)
            chi = self.randn(n, self.case["heads"], 4, 3).pow(2).sum(-1)
            k[:, :, self.outliers] = z / torch.sqrt(chi / 3.0) * 8.0
        else:
            k[:, :, self.outliers] *= 8.0
        return k.bfloat16()

    def values(self, n):
        return self.randn(n, self.case["heads"], D).bfloat16()


def _moment(q):
    """Second moment of Queries [n][H][D] in 64 bits, [H][D][D]."""
    x = q.permute(1, 0, 2).double()
    return x.transpose(1, 2) @ x / q.shape[0]


def _weights(M):
    dg = torch.diagonal(M, dim1=1, dim2=2)
    return dg / dg.mean(1, keepdim=True)


def _eig(M):
    """Eigenvalues in decreasing order, eigenvectors signed by their largest entry."""
    ev, vec = torch.linalg.eigh(M)
    ev, vec = ev.flip(1), vec.flip(2)
    top = vec.gather(1, vec.abs().argmax(1, keepdim=True))
    return ev, torch.where(top < 0, -vec, vec)


def _lloyd(x, C, iters):
    """Lloyd's k-means per head in 64 bits from strided tokens, [H][C][D] (sums of bf16 members are exact)."""
    x = x.permute(1, 0, 2).double()
    H, N, _ = x.shape
    cent = x[:, torch.arange(C, device=DEV) * N // C]
    for _ in range(iters):
        near = (cent.square().sum(2).unsqueeze(1) - 2.0 * (x @ cent.transpose(1, 2))).argmin(2)
        flat = (near + C * torch.arange(H, device=DEV).unsqueeze(1)).reshape(-1)
        tot = torch.zeros(H * C, D, dtype=torch.float64, device=DEV).index_add_(0, flat, x.reshape(-1, D))
        cnt = torch.bincount(flat, minlength=H * C).double().unsqueeze(1)
        cent = torch.where(cnt > 0, tot / cnt.clamp(min=1.0), cent.reshape(-1, D)).view(H, C, D)
    return cent


def _chunk(case, src, cold):
    """One finished chunk as the program holds it at the boundary: k, v, tables, w, U."""
    n, C, r = case["tokens"], case["centroids"], case["rank"]
    k, v = src.keys(n), src.values(n)
    kc, vc = (_lloyd(x, C, 2).bfloat16().contiguous() for x in (k, v))
    w = U = None
    if not cold:
        M = _moment(src.queries(1024))
        w = _weights(M).float().contiguous()
        if r:
            U = _eig(M)[1][:, :, :r].bfloat16().contiguous()
    return k, v, kc, vc, w, U


def _config(case):
    return qwm.config(case["heads"], case["centroids"], group_size=case["group"], psac_rank=case["rank"],
                      candidates=case["cands"], kmeans_iters=case["iters"], scale_format=int(case["two_level"]))


def _history(case, src):
    """The chunks appended before the call, the first one cold; a full window has lost its oldest chunk."""
    return (_chunk(case, src, cold=i == 0) for i in range(case["past"] + int(case["window"])))


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    cfg, src, op = _config(case), _Source(case, seed), case["op"]
    H, n, C = case["heads"], case["tokens"], case["centroids"]
    st = {"case": case, "cfg": cfg}
    if op == "attend":
        cache = qwm.Cache(cfg, n, case["past"], sliding_window=case["window"])
        for k, v, kc, vc, w, U in _history(case, src):
            qwm.qwm_quantize_append(cfg, cache, k, v, kc, vc, w=w, U=U)
        st["cache"], st["q"] = cache, src.queries(case["queries"])
        st["k"], st["v"] = (src.keys(case["cur"]), src.values(case["cur"])) if case["cur"] else (None, None)
        st["ws"] = qwm.attend_workspace(cfg, cache, case["queries"], case["cur"])
    elif op == "append":
        # a window of one chunk, so that each pass writes the same slot; what no pass writes is zero
        st["cache"] = qwm.Cache(cfg, n, 1, sliding_window=True)
        st["cache"].buffer.zero_()
        st["chunk"] = _chunk(case, src, cold=False)
    elif op == "fit":
        st["x"] = src.keys(n)
        st["out"] = torch.empty(H, C, D, dtype=torch.bfloat16, device=DEV)
        st["ws"] = torch.empty(qwm.qwm_fit_workspace_bytes(cfg, n), dtype=torch.uint8, device=DEV)
    elif op == "basis":
        st["q"], st["stats"] = src.queries(n), qwm.QueryStats(cfg)
    else:
        st["chunks"] = [(src.queries(n), src.keys(n), src.values(n)) for _ in range(case["past"])]
        st["ws"] = torch.empty(qwm.qwm_fit_workspace_bytes(cfg, n), dtype=torch.uint8, device=DEV)
    return st


def run(st):
    case, cfg, op = st["case"], st["cfg"], st["case"]["op"]
    if op == "attend":
        return qwm.qwm_attend(cfg, st["cache"], st["q"], st["k"], st["v"], want_lse=case["lse"], workspace=st["ws"])
    if op == "append":
        k, v, kc, vc, w, U = st["chunk"]
        qwm.qwm_quantize_append(cfg, st["cache"], k, v, kc, vc, w=w, U=U)
        return st["cache"].buffer
    if op == "fit":
        return qwm.qwm_fit_centroids(cfg, st["x"], centroids=st["out"], workspace=st["ws"])
    if op == "basis":
        st["stats"].reset()
        st["stats"].update(st["q"])
        w, U, ev = st["stats"].basis(eigenvalues=True)
        return [st["stats"].sums, w, ev] + ([U] if U is not None else [])
    # rollout: attend, then the chunk boundary, for each chunk of a new clip
    cache, stats = qwm.Cache(cfg, case["tokens"], case["past"]), qwm.QueryStats(cfg)
    outs, w, U = [], None, None
    for q, k, v in st["chunks"]:
        ws = qwm.attend_workspace(cfg, cache, case["tokens"], case["tokens"])
        outs.append(qwm.qwm_attend(cfg, cache, q, k, v, workspace=ws))
        kc = qwm.qwm_fit_centroids(cfg, k, workspace=st["ws"])
        vc = qwm.qwm_fit_centroids(cfg, v, workspace=st["ws"])
        qwm.qwm_quantize_append(cfg, cache, k, v, kc, vc, w=w, U=U)
        stats.update(q)
        w, U, _ = stats.basis()
        outs += [kc, vc, w] + ([U] if U is not None else [])
    return outs


def work(case):
    H, n, C, r, G = case["heads"], case["tokens"], case["centroids"], case["rank"], case["group"]
    scales = D // G + 2 if case["two_level"] else 2 * (D // G)
    packed = 2 * (D // 4 + scales + 2) + (r + 2 if r else 0)   # bytes of one token-head, Keys and Values
    tables = H * (2 * C * D * 2 + D * r * 2)

    def attend(nq, hist, cur):
        return {"bytes": H * hist * packed + -(-hist // n) * tables + 2 * H * D * 2 * (nq + cur),
                "flops": 2 * H * nq * (hist * (2 * D + r) + cur * 2 * D)}

    def append():
        return {"bytes": 2 * n * H * D * 2 + n * H * packed + 2 * tables + H * D * 4,
                "flops": 2 * 2 * n * H * C * D + 2 * n * H * D * r}

    def fit():
        return {"bytes": n * H * D * 2 + H * C * D * 2, "flops": 2 * n * H * C * D * case["iters"]}

    def basis():
        return {"bytes": n * H * D * 2 + H * D * D * 4 + 2 * H * D * 4 + H * D * r * 2,
                "flops": 2 * n * H * D * D + 9 * H * D ** 3}

    op = case["op"]
    if op == "attend":
        return attend(case["queries"], case["past"] * n, case["cur"])
    if op != "rollout":
        return {"append": append, "fit": fit, "basis": basis}[op]()
    parts = []
    for t in range(case["past"]):
        parts += [attend(n, t * n, n), append(), fit(), fit(), basis()]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------------------------ 64-bit results
def _half_up(x):
    """The smallest binary16 value >= x (x >= 0)."""
    h = x.half()
    return torch.where(h.double() < x, (h.view(torch.int16) + 1).view(torch.half), h).double()


def _rebuilt(case, x, tab, w, U):
    """What the cache holds for x [n][H][D]: centroid plus 2-bit residual, plus the PSAC correction, [H][n][D]."""
    G, ng, C = case["group"], D // case["group"], case["centroids"]
    x, mu = x.permute(1, 0, 2).double(), tab.double()
    H, n, _ = x.shape
    w = torch.ones(H, D, dtype=torch.float64, device=DEV) if w is None else w.double()
    wm = w.unsqueeze(1) * mu
    dist = (wm * mu).sum(2).unsqueeze(1) - 2.0 * (x @ wm.transpose(1, 2))
    cand = dist.topk(min(case["cands"], C), dim=2, largest=False).indices.sort(2).values
    wg, best = w.view(H, 1, ng, G).sum(3), None
    heads = torch.arange(H, device=DEV).unsqueeze(1)
    for m in range(cand.shape[2]):   # lowest QSAC score, ties to the lower index
        j = cand[:, :, m]
        res = (x - mu[heads, j]).view(H, n, ng, G)
        score = (wg * (res.amax(3) - res.amin(3)).square()).sum(2)
        if best is None:
            best, pick = score, j
        else:
            pick, best = torch.where(score < best, j, pick), torch.minimum(score, best)
    base = mu[heads, pick]
    res = (x - base).view(H, n, ng, G)
    lo, hi = res.amin(3).clamp(max=0.0), res.amax(3).clamp(min=0.0)
    s = (hi - lo) / 3.0
    if case["two_level"]:
        s2 = _half_up(s.amax(2, keepdim=True) / 255.0)
        s = torch.where(s2 > 0, torch.ceil(s / s2.clamp(min=1e-300)).clamp(max=255.0), torch.zeros_like(s)) * s2
    else:
        s = _half_up(s)
    inv = torch.where(s > 0, 1.0 / s.clamp(min=1e-300), torch.zeros_like(s)).unsqueeze(3)
    z = torch.round(-lo.unsqueeze(3) * inv).clamp(0, 3)
    out = base + (((torch.round(res * inv) + z).clamp(0, 3) - z) * s.unsqueeze(3)).view(H, n, D)
    if U is not None:
        U = U.double()
        err = x - out
        coef = err @ U
        sg = _half_up(coef.abs().amax(2, keepdim=True) / 127.0)
        fix = (torch.round(coef / sg.clamp(min=1e-300)).clamp(-127, 127) * sg) @ U.transpose(1, 2)
        keep = ((err - fix).square() @ w.unsqueeze(2)) < (err.square() @ w.unsqueeze(2))
        out = torch.where(keep, out + fix, out)
    return out


def exact(case, seed):
    src, op = _Source(case, seed), case["op"]
    if op == "attend":
        K, V = [], []
        for k, v, kc, vc, w, U in _history(case, src):
            K.append(_rebuilt(case, k, kc, w, U))
            V.append(_rebuilt(case, v, vc, None, None))
        K, V = K[-case["past"]:], V[-case["past"]:]
        q = src.queries(case["queries"]).permute(1, 0, 2).double()
        if case["cur"]:
            K.append(src.keys(case["cur"]).permute(1, 0, 2).double())
            V.append(src.values(case["cur"]).permute(1, 0, 2).double())
        out, lse = torch.empty_like(q), torch.empty(q.shape[:2], dtype=torch.float64, device=DEV)
        for h in range(q.shape[0]):
            kh, vh = torch.cat([x[h] for x in K]), torch.cat([x[h] for x in V])
            s = (q[h] @ kh.T).mul_(1.0 / math.sqrt(D))
            lse[h] = torch.logsumexp(s, 1)
            out[h] = s.sub_(lse[h].unsqueeze(1)).exp_() @ vh
        out = out.permute(1, 0, 2).contiguous()
        return (out, lse) if case["lse"] else out
    if op == "fit":
        return _lloyd(src.keys(case["tokens"]), case["centroids"], case["iters"])
    if op == "basis":
        q = src.queries(case["tokens"])
        M = _moment(q)
        ev, vec = _eig(M)
        return [M * q.shape[0], _weights(M), ev] + ([vec[:, :, :case["rank"]]] if case["rank"] else [])
    return None   # append returns bytes; the rollout's tables decide which bytes it attends over

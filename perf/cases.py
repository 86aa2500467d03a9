"""The measured cases: what a training program has this library do, once per
optimizer step and token table, through the public binding.

Three kinds of pass:
  dense   `Ember.step_dense`: W, r and c from a V x D fp32 gradient;
  sparse  `Ember.step_sparse`: the same from N token ids and one gradient row
          per occurrence;
  lmhead  `Ember.step_lmhead`: the head's gradient G = dlogits^T hidden over T
          tokens, formed by the library, then the step on it.

Inputs have the values of training: a token's gradient falls with its
frequency rank, token ids and targets follow Zipf(1.1), the errors of a head
are a softmax minus a one-hot over T.  The optimizer state is that of a run
that has taken T0 steps, and every pass is the next step of that run.
"""
import math

import torch

from paper_2607_01455_gb300.ember import Ember

LR = 1e-3
BETA2 = 0.999
EPS = 1e-8
T0 = 100          # steps taken before the first pass
SIGMA0 = 1e-3     # gradient scale of the most frequent token
ROW_STD = 1e-4    # gradient scale of one occurrence of a token
W_STD = 0.02
ZIPF = 1.1
LOGIT_STD = 2.0
MAX_ELEMS = 128256 * 8192
MAX_LM_WORK = 128256 * 8192 * 4096
MAX_SPARSE_ELEMS = 262144 * 768
DEVICE = "cuda"


def _dense(V, D, w, variant="full", zero=0.0, heavy=0.0, **kw):
    return dict(kind="dense", V=V, D=D, w=w, variant=variant, zero=zero, heavy=heavy, **kw)


def _sparse(V, D, N, w, ids, **kw):
    return dict(kind="sparse", V=V, D=D, N=N, w=w, ids=ids, **kw)


def _lmhead(V, D, T, w, **kw):
    return dict(kind="lmhead", V=V, D=D, T=T, w=w, **kw)


def listed():
    return [
        # a small table (a class head, a character vocabulary): the call is all latency
        _dense(1024, 64, "f32", name="dense_1024x64_f32"),
        # the smallest of the paper's tables, an odd number of rows, tied embedding and head
        _dense(50257, 768, "bf16", name="dense_50257x768_bf16"),
        # a tied table of a large vocabulary and a narrow model, with tokens never seen
        _dense(151936, 896, "bf16", zero=0.001, name="dense_tied_151936x896_bf16"),
        # a mid-size head whose weights are kept in 32 bits
        _dense(32000, 4096, "f32", name="dense_32000x4096_f32"),
        # the largest head, with heavy-tailed rows
        _dense(128256, 8192, "bf16", heavy=0.01, name="dense_128256x8192_bf16"),
        # a width that no vector access divides
        _dense(30011, 1003, "bf16", name="dense_ragged_30011x1003_bf16"),
        # the row-only ablation
        _dense(50304, 2048, "bf16", variant="row", name="dense_rowonly_50304x2048_bf16"),
        # an embedding step with a small batch (one sequence)
        _sparse(50257, 768, 1024, "bf16", "i64", name="sparse_50257x768_n1024"),
        # an embedding step of eight sequences of 4096 tokens over a large table
        _sparse(262144, 2048, 32768, "bf16", "i64", name="sparse_262144x2048_n32768"),
        # the paper's batch of 256 sequences of 1024 tokens
        _sparse(50257, 768, 262144, "bf16", "i32", name="sparse_50257x768_n262144"),
        # the head of a small model, gradient formed by the library
        _lmhead(50304, 768, 8192, "bf16", name="lmhead_50304x768_t8192"),
        # the largest head, gradient formed by the library
        _lmhead(128256, 8192, 4096, "bf16", name="lmhead_128256x8192_t4096"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "sparse", "sparse", "lmhead"])
    w = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if kind == "dense":
        D = _log(rng, 32, 12288)
        if rng.random() < 0.75:  # most widths are multiples of 16, some are any number
            D = max(32, D // 16 * 16)
        V = _log(rng, 512, max(512, min(260000, MAX_ELEMS // D)))
        variant = rng.choice(["full", "full", "full", "full", "row", "col"])
        return _dense(V, D, w, variant=variant, zero=rng.choice([0.0, 0.001]), heavy=rng.choice([0.0, 0.01]))
    if kind == "sparse":
        D = _log(rng, 64, 4096)
        if rng.random() < 0.85:
            D = max(64, D // 16 * 16)
        N = _log(rng, 128, min(262144, MAX_SPARSE_ELEMS // D))
        V = _log(rng, 2000, min(400000, MAX_ELEMS // D))
        return _sparse(V, D, N, w, rng.choice(["i64", "i32"]))
    D = max(128, _log(rng, 128, 8192) // 8 * 8)
    V = max(1024, _log(rng, 1024, min(160000, MAX_ELEMS // D)) // 8 * 8)
    T = _log(rng, 64, min(8192, MAX_LM_WORK // (V * D)))
    return _lmhead(V, D, T, w)


# ---- inputs, from the seed alone ----

def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed) * 1_000_003 + 17)


def _wtype(case):
    return torch.bfloat16 if case["w"] == "bf16" else torch.float32


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEVICE)


def _zipf_ids(g, V, n):
    cdf = torch.cumsum((torch.arange(V, device=DEVICE, dtype=torch.float64) + 1) ** -ZIPF, 0)
    u = torch.rand(n, generator=g, device=DEVICE, dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u, right=True).clamp_(max=V - 1)


def _inputs(case, seed):
    """(W, r, c, the arrays of the gradient), with the state T0 steps old."""
    g = _gen(seed)
    V, D = case["V"], case["D"]
    x = {}
    rank = torch.arange(V, device=DEVICE, dtype=torch.float64) + 1
    if case["kind"] == "dense":
        scale = (SIGMA0 * rank ** -0.5).float().unsqueeze(1)
        G = _randn(g, V, D).mul_(scale)
        nz, nh = round(case["zero"] * V), round(case["heavy"] * V)
        perm = torch.randperm(V, generator=g, device=DEVICE)
        heavy = perm[nz:nz + nh]
        if nh:  # Student's t with three degrees of freedom
            chi = sum(_randn(g, nh, D).square_() for _ in range(3))
            G[heavy] = _randn(g, nh, D) / torch.sqrt(chi / 3) * scale[heavy]
        if nz:
            G[perm[:nz]] = 0.0
        x["G"] = G
        row = scale.squeeze(1).double() ** 2
        if nz:
            row[perm[:nz]] = 0.0
    elif case["kind"] == "sparse":
        ids = _zipf_ids(g, V, case["N"])
        x["rows"] = _randn(g, case["N"], D).mul_(ROW_STD)
        x["ids"] = ids if case["ids"] == "i64" else ids.to(torch.int32)
        p = rank ** -ZIPF
        row = ROW_STD ** 2 * case["N"] * p / p.sum()
    else:
        T = case["T"]
        y = _zipf_ids(g, V, T)
        x["dlogits"] = torch.empty(T, V, device=DEVICE, dtype=torch.bfloat16)
        for t in range(0, T, 512):
            q = torch.softmax(_randn(g, min(512, T - t), V).mul_(LOGIT_STD), dim=1)
            q[torch.arange(q.shape[0], device=DEVICE), y[t:t + 512]] -= 1.0
            x["dlogits"][t:t + 512] = q / T
        x["hidden"] = _randn(g, T, D).to(torch.bfloat16)
        p = rank ** -ZIPF
        row = p / p.sum() / T
    W = _randn(g, V, D).mul_(W_STD).to(_wtype(case))
    taken = 1.0 - BETA2 ** T0  # what a moment of T0 steps has reached of its mean
    r = (row * taken * (0.5 + torch.rand(V, generator=g, device=DEVICE))).float()
    c = (row.mean() * taken * (0.5 + torch.rand(D, generator=g, device=DEVICE))).float()
    return W, r, c, x


def prepare(case, seed):
    W, r, c, x = _inputs(case, seed)
    emb = Ember(case["V"], case["D"], wdtype=case["w"], beta2=BETA2, eps=EPS, variant=case.get("variant", "full"),
                max_sparse_N=case.get("N", 0), device=DEVICE)
    emb.r.copy_(r)
    emb.c.copy_(c)
    out = {"W": W, "r": emb.r, "c": emb.c}
    if case["kind"] == "lmhead":
        x["G"] = out["G"] = torch.empty(case["V"], case["D"], device=DEVICE)
    return {"kind": case["kind"], "emb": emb, "W": W, "x": x, "t": T0, "out": out}


def run(state):
    state["t"] += 1
    emb, W, x = state["emb"], state["W"], state["x"]
    if state["kind"] == "dense":
        emb.step_dense(W, x["G"], LR, state["t"])
    elif state["kind"] == "sparse":
        emb.step_sparse(W, x["ids"], x["rows"], LR, state["t"])
    else:
        emb.step_lmhead(W, x["dlogits"], x["hidden"], x["G"], LR, state["t"])
    return state["out"]


def _distinct(V, N):
    """Distinct ids to be expected among N draws of Zipf(1.1) over [0, V)."""
    p = (torch.arange(V, dtype=torch.float64) + 1) ** -ZIPF
    return float((1 - torch.exp(N * torch.log1p(-p / p.sum()))).sum())


def work(case):
    V, D = case["V"], case["D"]
    w = 2 if case["w"] == "bf16" else 4
    state = 8 * (V + D)  # r and c, read and written
    if case["kind"] == "dense":
        return {"bytes": 4 * V * D + 2 * w * V * D + state, "flops": 10 * V * D}
    if case["kind"] == "sparse":
        N, U = case["N"], _distinct(V, case["N"])
        idb = 8 if case["ids"] == "i64" else 4
        return {"bytes": 4 * N * D + idb * N + 2 * w * U * D + state, "flops": (N + 10 * U) * D}
    T = case["T"]
    return {"bytes": 2 * T * (V + D) + 4 * V * D + 2 * w * V * D + state, "flops": 2 * V * D * T + 10 * V * D}


def tolerance(case):
    """Of W, r, c (and the head's G) together, about four times what one
    correct implementation is off the 64-bit step.  A bf16 weight next to a
    rounding boundary may round either way (seen on up to 1e-5 of the weights,
    1e-4 of a head's): one bf16 ulp, at most 2^-7 of the value.  The head's G
    is a sum of T bf16 products on the tensor cores, whose 32-bit additions
    truncate (1e-5 at T = 8192); the other sums are off by 5e-8 at most."""
    head = case["kind"] == "lmhead"
    if case["w"] == "bf16":
        return {"rel": 6e-5 if head else 2e-5, "max": 1.6e-2}
    return {"rel": 4e-5, "max": 3e-3} if head else {"rel": 1e-6, "max": 4e-6}


def exact(case, seed):
    """The step in 64 bits: Algorithm 1 on the same inputs (W not rounded)."""
    W, r, c, x = _inputs(case, seed)
    V, D = case["V"], case["D"]
    variant = case.get("variant", "full")
    r, c = r.double(), c.double()
    chunk = max(1, (1 << 27) // D)
    out = {}
    if case["kind"] == "sparse":
        uniq, inv = torch.unique(x["ids"].long(), return_inverse=True)
        S = torch.zeros(uniq.numel(), D, device=DEVICE, dtype=torch.float64)
        step = max(1, (1 << 26) // D)
        for n in range(0, case["N"], step):
            S.index_add_(0, inv[n:n + step], x["rows"][n:n + step].double())
        rows_of = [(uniq, S)]
    elif case["kind"] == "dense":
        G = x["G"]
        rows_of = [(slice(v, min(V, v + chunk)), None) for v in range(0, V, chunk)]
    else:
        h = x["hidden"].double()
        G = torch.empty(V, D, device=DEVICE, dtype=torch.float64)
        for v in range(0, V, 8192):
            G[v:v + 8192] = x["dlogits"][:, v:v + 8192].double().T @ h
        out["G"] = G
        rows_of = [(slice(v, min(V, v + chunk)), None) for v in range(0, V, chunk)]
    rsq = torch.zeros(V, device=DEVICE, dtype=torch.float64)
    csq = torch.zeros(D, device=DEVICE, dtype=torch.float64)
    for at, g in rows_of:
        g2 = (G[at].double() if g is None else g).square()
        rsq[at] = g2.sum(1)
        csq += g2.sum(0)
    r = BETA2 * r + (1 - BETA2) * rsq / D
    c = BETA2 * c + (1 - BETA2) * csq / V
    bc = 1 - BETA2 ** (T0 + 1)
    rh, ch = r / bc, c / bc
    s = torch.sqrt(rh.mean() * ch.mean())
    W = W.double()
    for at, g in rows_of:
        g = G[at].double() if g is None else g
        if variant == "row":
            v = rh[at].unsqueeze(1).expand(-1, D)
        elif variant == "col":
            v = ch.unsqueeze(0).expand(g.shape[0], -1)
        else:
            v = rh[at].unsqueeze(1) * (ch / s)
        W[at] = W[at] - LR * g / (torch.sqrt(v) + EPS)
    out.update(W=W, r=r, c=c)
    return out

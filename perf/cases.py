"""The timed cases of the ELSAA attention operator: what they run, on which
inputs, the work each cannot do without, and its result in 64 bits.

A case is one attention layer over all heads of a batch, called through the
public binding (paper_2607_20214_gb300.elsaa) with a workspace that the caller
keeps, as a layer of a user's model does. Sizes come from the repository's
workloads (c1-c5, c3 causal) and its tests; the others fill the range between
them: one short prompt, ragged lengths, the smallest and the largest batch.

kinds: forward  elsaa_forward (sorted blocks)
       gated    elsaa_forward_gated (gate MLP and lambda_i in the call)
       topk     elsaa_forward with the per-query top-k selector
       causal   elsaa_forward with causal = 1
       train    elsaa_forward (orders kept), elsaa_forward_race_summaries,
                elsaa_backward
"""
from __future__ import annotations

import math

import torch

from paper_2607_20214_gb300 import elsaa as E

_DEFAULTS = dict(kind="forward", B=1, H=1, N=1024, d=64, dtype="bf16", b=64,
                 L=8, sort_bits=5, temp="plain", aux=False, gates=False,
                 neighbors=0, k=0, c=1, base=4096, hidden=64)


def _case(**kw):
    return dict(_DEFAULTS, **kw)


def listed():
    return [
        # smallest call: one fp32 head (the workload that is checked in
        # full against the oracle); launches and latency decide
        _case(name="fp32_small", dtype="fp32", B=1, H=1, N=1024, d=64, b=32,
              L=4),
        # one short bf16 sequence through a 12-head layer: latency
        _case(name="bf16_short", B=1, H=12, N=1024, d=64, b=64, L=8),
        # an odd batch of image-like token counts: 75 blocks of 64, so the
        # last 128-row tile of every head is half empty; 4 sort bits
        _case(name="ragged", B=3, H=5, N=4800, d=128, b=64, L=8,
              sort_bits=4),
        # a batch of mid-length sequences, heads of mixed temperature; the
        # log denominators and the multiplier are read back as well, as by a
        # model that logs its branch masses
        _case(name="mid_batch", B=4, H=12, N=4096, d=64, b=64, L=8,
              temp="cycle", aux=True),
        # the headline configuration: prefill at N = 16K, d_h = 128
        _case(name="prefill_16k", B=2, H=16, N=16384, d=128, b=128, L=16,
              temp="uniform"),
        # long context: N = 64K, 256 keys per query; the largest call
        _case(name="long_64k", B=1, H=32, N=65536, d=128, b=256, L=16),
        # the headline with the learned gates and lambda_i in the call
        _case(name="gated_16k", kind="gated", B=2, H=16, N=16384, d=128,
              b=128, L=16, temp="uniform"),
        # the headline with the per-query top-k selector
        _case(name="topk_16k", kind="topk", B=2, H=16, N=16384, d=128,
              b=128, L=16, temp="uniform", k=128, c=2),
        # a short causal prompt with the smaller base segment (256 rows)
        _case(name="causal_2k", kind="causal", B=1, H=8, N=2048, d=64, b=64,
              L=8, base=256),
        # causal prefill at N = 16K with 4096-row base segments
        _case(name="causal_16k", kind="causal", B=2, H=16, N=16384, d=128,
              b=128, L=16, temp="uniform", base=4096),
        # a small training step with learned gates and per-token lambda:
        # their gradients are returned too
        _case(name="train_small", kind="train", B=2, H=8, N=1024, d=64, b=64,
              L=4, gates=True),
        # the training workload: forward and backward, B = 8, N = 8192
        _case(name="train_8k", kind="train", B=8, H=12, N=8192, d=64, b=64,
              L=8, temp="two"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: kinds, types, head sizes, block sizes and
    ranks as in the listed ones; B, H and N spread over their logarithms, N
    any multiple of the block (of 128 rows times a power of two in the causal
    recursion)."""
    kind = rng.choice(["forward", "forward", "forward", "gated", "topk",
                       "causal", "train"])
    d = rng.choice([64, 128])
    kw = dict(kind=kind, d=d, sort_bits=rng.choice([4, 5]),
              temp=rng.choice(["plain", "two", "cycle", "uniform"]))
    # token-heads x d of one call, at most the largest of its kind
    cap = dict(forward=32 * 65536 * 128, gated=32 * 16384 * 128,
               topk=32 * 16384 * 128, causal=32 * 16384 * 128,
               train=96 * 8192 * 64)[kind]
    if kind == "forward" and rng.random() < 0.25:  # fp32: small calls
        kw.update(dtype="fp32", d=64, b=32, L=4, aux=rng.random() < 0.5)
        cap, d = 12 * 4096 * 64, 64
    elif kind == "train":
        kw.update(d=64, b=64, L=rng.choice([4, 8]), gates=rng.random() < 0.5)
        d = 64
    elif kind == "topk":
        kw.update(b=128, c=rng.choice([2, 3]), L=rng.choice([4, 8, 16]))
        kw["k"] = rng.randrange(64, kw["c"] * 128 + 1)
    elif kind == "causal":
        kw.update(b=rng.choice([64, 128]), L=rng.choice([4, 8, 16]),
                  base=rng.choice([256, 1024, 4096]))
    else:
        kw.update(b=rng.choice([32, 64, 128, 256]),
                  L=rng.choice([4, 8, 16]) if d == 128 else
                  rng.choice([4, 8]))
        if kind == "forward":
            kw["aux"] = rng.random() < 0.25
            kw["gates"] = rng.random() < 0.25
            if kw["b"] == 128:
                kw["neighbors"] = rng.choice([0, 0, 1])
        else:
            kw["hidden"] = rng.choice([64, 128])
    heads_cap = 96 if kind in ("forward", "train") else 32
    total = _log_int(rng, 1, heads_cap)
    B = max(1, min(8, _log_int(rng, 1, 8)))
    H = max(1, total // B)
    top_n = min(65536 if kind == "forward" else 16384, cap // (B * H * d))
    step = kw.get("b", 64)
    if kind == "train":
        step = 128
    low = max(4 * step, 512)
    n = _log_int(rng, min(low, top_n), top_n)
    if kind == "causal":
        lv = 0
        while n / (1 << lv) > kw["base"]:
            lv += 1
        step = 128 << lv
        n = min(n, kw["base"] << lv)
    n = max(step, n // step * step)
    if kind == "topk":
        n = max(n, kw["c"] * 128)
    return _case(B=B, H=H, N=n, **kw)


# ------------------------------------------------------------------- inputs

def _temps(case, device):
    H = case["H"]
    if case["temp"] == "cycle":
        return torch.tensor([(0.5, 1.0, 2.0, 4.0)[h % 4] for h in range(H)],
                            device=device)
    if case["temp"] == "uniform":
        return torch.linspace(0.5, 4.0, H, device=device)
    return torch.full((H,), 2.0 if case["temp"] == "two" else 1.0,
                      device=device)


def _inputs(case, seed, device="cuda"):
    """Q, K, V ~ N(0, 1) with per-head query temperatures; with mixed
    temperatures one query in eight of the even heads finds eight keys close
    to it (needles); in sequences of 32K and more every 64th key is repeated
    half a sequence later. Planes are Gaussian, RACE planes and the gate
    network's first layer bf16-representable."""
    B, H, N, d = (case[x] for x in ("B", "H", "N", "d"))
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=device)

    def bf(x):
        return x.to(torch.bfloat16).float()

    q, k, v = randn(B, H, N, d), randn(B, H, N, d), randn(B, H, N, d)
    if case["temp"] == "cycle" and N >= 4096 and case["kind"] == "forward":
        src = torch.arange(N, device=device) // 8 * 8
        for h in range(0, H, 2):
            pi = torch.randperm(N, generator=g, device=device)
            k[:, h, pi] = q[:, h, src] + 0.1 * randn(B, N, d)
    if N >= 32768:
        m = torch.arange(N // 128, device=device) * 64
        k[:, :, N // 2 + m] = k[:, :, m]
    q *= _temps(case, device).view(1, H, 1, 1)
    t = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    x = dict(q=q.to(t), k=k.to(t), v=v.to(t),
             w_sort=randn(H, case["sort_bits"], d),
             w_race=bf(randn(H, case["L"], 4, d)))
    if case["gates"]:
        x["gates"] = torch.sigmoid(randn(B, H, N, 2))
        x["lam"] = 0.3 + torch.sigmoid(0.5 * randn(B, H, N))
    if case["kind"] == "gated":
        n = case["hidden"]
        x["mlp"] = dict(
            hidden=n, w1=bf(randn(H, n, d) / d ** 0.5), b1=0.1 * randn(H, n),
            w2=randn(H, 2, n) / n ** 0.5, b2=0.5 * randn(H, 2),
            w_lambda=bf(0.05 * randn(H, d)),
            b_lambda=torch.zeros(H, device=device),
            c_lambda=torch.full((H,), 0.3, device=device), lambda_min=1e-6)
    if case["kind"] == "train":
        x["do"] = randn(B, H, N, d).to(t)
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    p = E.make_params(
        case["B"], case["H"], case["N"], case["d"], dtype=case["dtype"],
        block_size=case["b"], sort_bits=case["sort_bits"],
        race_tables=case["L"], causal=int(kind == "causal"),
        causal_base_len=case["base"], neighbor_blocks=case["neighbors"],
        selector=int(kind == "topk"), topk=case["k"],
        topk_blocks=case["c"])
    s = dict(x, case=case, p=p)

    def scratch(n):
        return torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")

    if kind == "gated":
        s["ws"] = scratch(E.elsaa_forward_gated_workspace_size(p, x["mlp"]))
    else:
        s["ws"] = scratch(E.elsaa_workspace_size(p))
    if kind == "train":
        s["bws"] = scratch(E.elsaa_backward_workspace_size(p))
    return s


def run(s):
    case, p = s["case"], s["p"]
    shape = (case["B"], case["H"], case["N"])
    qkv = (s["q"], s["k"], s["v"], s["w_sort"], s["w_race"])

    def new(dtype, *more):
        return torch.empty(shape + more, dtype=dtype, device="cuda")

    if case["kind"] == "gated":
        return dict(o=E.elsaa_forward_gated(p, s["mlp"], *qkv,
                                            workspace=s["ws"]))
    tok = dict(lambda_tok=s.get("lam"), gates=s.get("gates"))
    if case["kind"] == "train":
        pq, pk = new(torch.int32), new(torch.int32)
        o = E.elsaa_forward(p, *qkv, perm_q=pq, perm_k=pk, workspace=s["ws"],
                            **tok)
        A, Bm = E.elsaa_forward_race_summaries(p, s["ws"])
        if case["gates"]:
            tok.update(d_gates=new(torch.float32, 2),
                       d_lambda=new(torch.float32))
        dq, dk, dv = E.elsaa_backward(p, *qkv, s["do"], pq, pk, race_A=A,
                                      race_B=Bm, workspace=s["bws"], **tok)
        out = dict(o=o, perm_q=pq, perm_k=pk, dq=dq, dk=dk, dv=dv)
        if case["gates"]:
            out.update(d_gates=tok["d_gates"], d_lambda=tok["d_lambda"])
        return out
    out = {}
    if case["aux"]:
        out = dict(log_d_sparse=new(torch.float32), d_lr=new(torch.float32),
                   m_sparse=new(torch.float32))
    out["o"] = E.elsaa_forward(p, *qkv, workspace=s["ws"], **tok, **out)
    return out


# --------------------------------------------------------------------- work

def work(case):
    """Inputs read once, outputs written once; the multiply-adds of the
    definitions (2 per product), per token and head."""
    B, H, N, d, b, L = (case[x] for x in ("B", "H", "N", "d", "b", "L"))
    r = 16 * L
    elt = 4 if case["dtype"] == "fp32" else 2
    tok = B * H * N
    nbytes = 4 * d * elt + (12 if case["aux"] else 0)
    nbytes += 12 if case["gates"] else 0
    keys = b
    if case["kind"] == "causal":
        leaf, lv = N, 0
        while leaf > case["base"]:
            leaf, lv = leaf // 2, lv + 1
        keys = (leaf + 1) / 2 + lv * b / 2
    elif case["kind"] == "topk":
        keys = case["k"]
    elif case["neighbors"]:
        keys = 3 * b - 2 * b * b / N
    flops = 4 * keys * d + 4 * r * (d + 1) + 16 * d * L
    flops += 4 * d * case["sort_bits"]
    if case["kind"] == "topk":
        flops += 2 * d * case["c"] * b
    if case["kind"] == "gated":
        flops += 2 * (case["hidden"] + 1) * d + 4 * case["hidden"]
    if case["kind"] == "train":
        # q, k, v, dO read again for the gradients, three fp32 gradients
        # and two orders written; five block products, four of features
        nbytes += 4 * d * elt + 3 * d * 4 + 8 + (12 if case["gates"] else 0)
        flops += 10 * b * d + 12 * r * d + 24 * d * L
    weights = H * (case["sort_bits"] + 4 * L) * d * 4
    return {"bytes": tok * nbytes + weights, "flops": tok * flops}


# -------------------------------------------------------------- 64-bit result

def _chain(x, w):
    """<w, x> as the sequential fp32 fused multiply-add chain that defines
    the hash bits and the selection scores (products exact in 64 bits, one
    rounding to 32 bits per step). x [..., d], w [..., d], broadcast."""
    acc = None
    for i in range(x.shape[-1]):
        p = x[..., i].double() * w[..., i].double()
        acc = (p if acc is None else p + acc.double()).float()
    return acc


def _order(x, w):
    """The stable order of the rows by the Gray rank of their sign codes."""
    code = torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
    for p in range(w.shape[0]):
        bit = _chain(x.float(), w[p].float()) > 0
        code |= bit.long() << p
    rank = code.clone()
    for s in (1, 2, 4):
        rank ^= rank >> s
    return torch.argsort(rank, stable=True), rank


def _phi(x, w, beta=1.0):
    """RACE features, [n, L, 16]: softmax over the corners of tanh(W x)."""
    L, g, d = w.shape
    u = torch.tanh(x @ w.reshape(L * g, d).T).reshape(-1, L, g)
    s = torch.sigmoid(2 * beta * u)
    out = torch.ones(u.shape[:2] + (1,), dtype=u.dtype, device=u.device)
    for bit in range(g):  # bit of the bucket index: the later the higher
        out = torch.cat([out * (1 - s[..., bit:bit + 1]),
                         out * s[..., bit:bit + 1]], -1)
    return out


def _attend(z, v, eps):
    """(O, log d) of one softmax block: O = sum e^z v / (sum e^z + eps)."""
    top = z.amax(-1, keepdim=True)
    e = torch.exp(z - top)
    s = e.sum(-1, keepdim=True)
    return e @ v / (s + eps * torch.exp(-top)), (top + torch.log(s))[..., 0]


def _blocks(q, k, v, pq, pk, b, eps, nb=0):
    N, d = q.shape
    T = N // b
    qs, ks, vs = (x[i].reshape(T, b, d) for x, i in ((q, pq), (k, pk),
                                                     (v, pk)))
    z, vv = [], []
    for o in range(-nb, nb + 1):
        t = torch.arange(T, device=q.device) + o
        inside = (t >= 0) & (t < T)
        t = t.clamp(0, T - 1)
        s = qs @ ks[t].transpose(1, 2) / math.sqrt(d)
        z.append(s.masked_fill(~inside.view(T, 1, 1), -math.inf))
        vv.append(vs[t])
    os, ls = _attend(torch.cat(z, -1), torch.cat(vv, 1), eps)
    inv = torch.argsort(pq)
    return os.reshape(N, d)[inv], ls.reshape(N)[inv]


def _topk(q, k, v, pq, pk, case, eps):
    """Candidate blocks by the scores of fp32 block sums, then the k keys of
    largest score per query (ties: lower index), then the block step."""
    N, d = q.shape
    b, c, kk = case["b"], case["c"], case["k"]
    T = N // b
    qs, ks = q[pq].reshape(T, b, d), k[pk].reshape(T, b, d)
    sums = []
    for x in (qs, ks):
        acc = torch.zeros(T, d, dtype=torch.float32, device=q.device)
        for i in range(b):
            acc = acc + x[:, i].float()
        sums.append(acc)
    score = _chain(sums[0][:, None], sums[1][None])
    own = torch.arange(T, device=q.device)
    score[own, own] = math.inf
    cand = torch.sort(score, dim=1, descending=True,
                      stable=True)[1][:, :c]
    kid = pk.reshape(T, b)[cand].reshape(T, c * b)
    kid = torch.sort(kid, 1)[0]  # by index: a stable sort breaks ties low
    os = torch.empty(T, b, d, dtype=q.dtype, device=q.device)
    step = 16
    for t in range(0, T, step):
        kt = k[kid[t:t + step]]
        sc = _chain(qs[t:t + step].float()[:, :, None], kt.float()[:, None])
        at = torch.sort(sc, dim=2, descending=True, stable=True)[1][..., :kk]
        z = qs[t:t + step] @ kt.transpose(1, 2) / math.sqrt(d)
        keep = torch.zeros_like(z, dtype=torch.bool).scatter_(2, at, True)
        os[t:t + step] = _attend(z.masked_fill(~keep, -math.inf),
                                 v[kid[t:t + step]], eps)[0]
        if t == 0:
            ls = torch.empty(T, b, dtype=q.dtype, device=q.device)
        ls[t:t + step] = torch.logsumexp(z.masked_fill(~keep, -math.inf), -1)
    inv = torch.argsort(pq)
    return os.reshape(N, d)[inv], ls.reshape(N)[inv]


def _causal_sparse(q, k, v, hq, hk, case, eps):
    n, d = q.shape
    if n <= case["base"]:
        z = q @ k.T / math.sqrt(d)
        z = z.masked_fill(torch.ones_like(z, dtype=torch.bool).triu(1),
                          -math.inf)
        return _attend(z, v, eps)
    m = n // 2
    o1, l1 = _causal_sparse(q[:m], k[:m], v[:m], hq[:m], hk[:m], case, eps)
    o2, l2 = _causal_sparse(q[m:], k[m:], v[m:], hq[m:], hk[m:], case, eps)
    o3, l3 = _blocks(q[m:], k[:m], v[:m], torch.argsort(hq[m:], stable=True),
                     torch.argsort(hk[:m], stable=True), case["b"], eps)
    mu = torch.maximum(l2, l3)
    w2, w3 = torch.exp(l2 - mu), torch.exp(l3 - mu)
    s = w2 + w3 + eps
    o2 = (w2[:, None] * o2 + w3[:, None] * o3) / s[:, None]
    return torch.cat([o1, o2]), torch.cat([l1, mu + torch.log(s)])


def _causal_race(fq, fk, v, L):
    """(Num, Den) over the keys up to each query's own, 128 at a time."""
    n, d = v.shape
    a = fq.reshape(n // 128, 128, -1)
    f = fk.reshape(n // 128, 128, -1)
    v1 = torch.cat([v, torch.ones_like(v[:, :1])], 1).reshape(-1, 128, d + 1)
    state = torch.cumsum(f.transpose(1, 2) @ v1, 0)
    past = torch.cat([torch.zeros_like(state[:1]), state[:-1]])
    out = (a @ past + (a @ f.transpose(1, 2)).tril() @ v1) / L
    out = out.reshape(n, d + 1)
    return out[:, :d], out[:, d]


def _head(case, q, k, v, wr, lam, gs, gl, orders, eps=1e-6):
    """One head: (O, log d_sparse, d_lr, m) in the type of q."""
    kind, L = case["kind"], case["L"]
    (pq, hq), (pk, hk) = orders
    fq, fk = _phi(q, wr).flatten(1), _phi(k, wr).flatten(1)
    if kind == "causal":
        os, ls = _causal_sparse(q, k, v, hq, hk, case, eps)
        num, den = _causal_race(fq, fk, v, L)
    else:
        if kind == "topk":
            os, ls = _topk(q, k, v, pq, pk, case, eps)
        else:
            os, ls = _blocks(q, k, v, pq, pk, case["b"], eps,
                             case["neighbors"])
        num, den = fq @ (fk.T @ v) / L, fq @ fk.sum(0) / L
    olr = num / (den + eps)[:, None]
    # d_s / (d_s + lambda d_lr + eps), in logarithms
    m = torch.sigmoid(ls - torch.log(lam * den + eps))
    o = (gs * m)[:, None] * os + gl[:, None] * olr
    return o, ls, den, m


def _gate_net(mlp, h, q):
    a = q @ mlp["w1"][h].double().T + mlp["b1"][h].double()
    a = a * torch.sigmoid(a)
    g = torch.sigmoid(a @ mlp["w2"][h].double().T + mlp["b2"][h].double())
    lam = mlp["c_lambda"][h].double() + torch.sigmoid(
        q @ mlp["w_lambda"][h].double() + mlp["b_lambda"][h].double())
    return lam.clamp_min(mlp["lambda_min"]), g[:, 0], g[:, 1]


def exact(case, seed):
    """run()'s outputs in 64 bits, head by head, from plain torch."""
    x = _inputs(case, seed)
    kind = case["kind"]
    B, H, N = case["B"], case["H"], case["N"]
    train = kind == "train"
    names = ["dq", "dk", "dv"] if train else []
    if train and case["gates"]:
        names += ["d_gates", "d_lambda"]
    if case["aux"]:
        names += ["log_d_sparse", "d_lr", "m_sparse"]
    shapes = dict(o=x["q"].shape, dq=x["q"].shape, dk=x["q"].shape,
                  dv=x["q"].shape, d_gates=(B, H, N, 2))
    out = {n: torch.empty(shapes.get(n, (B, H, N)), dtype=torch.float64,
                          device="cuda") for n in ["o"] + names}
    for i in range(B):
        for h in range(H):
            q, k, v = (x[n][i, h].double() for n in "qkv")
            orders = [_order(x[n][i, h], x["w_sort"][h]) for n in "qk"]
            if kind == "gated":
                lam, gs, gl = _gate_net(x["mlp"], h, q)
            elif case["gates"]:
                lam = x["lam"][i, h].double()
                gs, gl = x["gates"][i, h].double().unbind(-1)
            else:
                lam = gs = gl = torch.ones(N, dtype=torch.float64,
                                           device="cuda")
            at = [q, k, v, gs, gl, lam]
            if train:
                at = [t.detach().clone().requires_grad_() for t in at]
            q, k, v, gs, gl, lam = at
            o, ls, den, m = _head(case, q, k, v,
                                  x["w_race"][h].double(), lam, gs, gl,
                                  orders)
            out["o"][i, h] = o.detach()
            if case["aux"]:
                out["log_d_sparse"][i, h] = ls
                out["d_lr"][i, h] = den
                out["m_sparse"][i, h] = m
            if train:
                gr = torch.autograd.grad(o, at, x["do"][i, h].double())
                for n, t in zip(("dq", "dk", "dv"), gr):
                    out[n][i, h] = t
                if case["gates"]:
                    out["d_gates"][i, h] = torch.stack(gr[3:5], -1)
                    out["d_lambda"][i, h] = gr[5]
    if train:
        out.update(perm_q=None, perm_k=None)
    return out

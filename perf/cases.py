"""What this framework's performance is measured on: its public calls over the range that a program has them do.

Four kinds of case, each one call:
  stack    ``stack_forward``: the pruned stack of attention layers on device tensors (the main path)
  host     ``stack_forward_host``: the same stack on page-locked host tensors
  layer    ``layer_forward``: one attention + pruning layer on tokens in current order
  encoder  ``encoder_layer_forward``: one whole encoder layer (projections, attention with pruning, feed-forward)

Inputs follow the generator of the repository's workloads: Q, K, V ~ N(0, 1) in bf16, a share of salient tokens
whose key rows are scaled up, token 0 and a few further positions global.  A token whose score lies within 1e-4 / n
of the keep threshold has its Q and K rows drawn again, as in the repository's parity fixtures: the kept lists are
whole numbers, and every correct implementation takes the same decision.  The decisions come from a plain 64-bit
evaluation in torch (``_attention``), which ``exact`` uses as well.
"""
from __future__ import annotations

import functools
import math

import torch

import paper_2310_07109_gb300 as sc

HEAD = 64
MARGIN = 1e-4      # of the mean score 1 / n
RELATIVE, ABSOLUTE, TOP_RATIO = 0, 1, 2


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _stack(name, B, L, w, *, kind="stack", layers=12, H=12, extra=0, frac=0.10, scale=3.0, a0=0.3, a1=0.9,
           rule=RELATIVE, ragged=1.0):
    """``extra``: global positions beside token 0; ``frac``/``scale``: salient tokens; ``a0`` to ``a1``: the keep
    rule's value, linear in depth; ``ragged``: true lengths uniform in [ragged L, L], the rest padding."""
    return dict(name=name, kind=kind, layers=layers, B=B, L=L, H=H, w=w, extra=extra, frac=frac, scale=scale,
                a0=a0, a1=a1, rule=rule, ragged=ragged)


def listed():
    return [
        # one short function scanned on its own (an editor plug-in): latency only
        _stack("stack_one_short", 1, 96, 64),
        # a batch of short functions, padded to the longest: the bulk of the paper's length distribution
        _stack("stack_batch_short", 16, 333, 64, ragged=0.4),
        # the RoBERTa-base shaped stack at the paper's max_length
        _stack("stack_1024", 8, 1024, 256),
        # longer functions of differing true length: padding removal, then the pruned stack
        _stack("stack_2048_ragged", 4, 2048, 256, ragged=0.5),
        # the longest inputs, with eight special tokens beside CLS (bench.py's default workload)
        _stack("stack_4096_globals", 2, 4096, 256, extra=8, frac=0.05, scale=4.0, a0=0.4, a1=1.0),
        # the paper's sparse-attention model without token pruning (its control), narrow window and mid length
        _stack("stack_unpruned_w64", 3, 1000, 64, a0=0.0, a1=0.0),
        # the same control at full length: the largest case
        _stack("stack_unpruned_4096", 4, 4096, 256, a0=0.0, a1=0.0),
        # the top-k family of pruning rules: a fixed share of the tokens goes at each layer
        _stack("stack_top_ratio", 4, 777, 128, extra=2, a0=0.95, a1=0.8, rule=TOP_RATIO),
        # Q, K, V and the results in host memory (a service whose encoder front end runs elsewhere)
        _stack("host_1024", 4, 1024, 256, kind="host"),
        # one layer with the widest window on ragged, already compacted tokens: a layer-by-layer caller
        _stack("layer_w512", 2, 3000, 512, kind="layer", layers=1, extra=15, a0=0.7, a1=0.7, ragged=0.6),
        # one encoder layer as in the RoBERTa-base shaped model, a full batch
        _stack("encoder_1024", 8, 1024, 256, kind="encoder", layers=1),
        # ... and the batch of one short function
        _stack("encoder_one_short", 1, 200, 64, kind="encoder", layers=1),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stack"] * 6 + ["host", "layer", "layer", "encoder", "encoder"])
    L = _log_uniform(rng, 48, 4096)
    B = max(1, min(32, _log_uniform(rng, L, 8192) // L))
    H = rng.choice([12, 12, 12, 4, 16 if B * L <= 6144 else 8])
    w = _log_uniform(rng, 16, 512 if kind == "layer" or L <= 1024 else 300)
    extra = min(L // 8, rng.choice([0, 0, 1, 3, 8, 15]))
    frac, scale = rng.choice([(0.10, 3.0), (0.05, 4.0)])
    ragged = rng.choice([1.0, 1.0, 0.5, 0.8])
    layers = 1 if kind in ("layer", "encoder") else rng.choice([12, 12, 12, 6])
    rule, a0, a1 = rng.choice([(RELATIVE, 0.3, 0.9), (RELATIVE, 0.4, 1.0), (RELATIVE, 0.2, 0.7), (RELATIVE, 0.0, 0.0),
                               (ABSOLUTE, 0.01 / 12, 0.01), (TOP_RATIO, 0.95, 0.8)])
    c = _stack("", B, L, w, kind=kind, layers=layers, H=H, extra=extra, frac=frac, scale=scale, a0=a0, a1=a1, rule=rule,
               ragged=ragged)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
def _attention(q, k, v, w, gl):
    """q, k, v float64 [n, H, 64], gl the current indices of the global tokens: (O [n, H, 64], scores [n])."""
    n, H, _ = q.shape
    q, k, v = (t.transpose(0, 1) for t in (q, k, v))
    at = torch.arange(n, device=q.device)
    glob = torch.zeros(n, dtype=torch.bool, device=q.device)
    glob[gl] = True
    O, s = torch.empty_like(q), torch.zeros(n, dtype=torch.float64, device=q.device)
    for i0 in range(0, n, 512):
        i1 = min(n, i0 + 512)
        lo, hi = max(0, i0 - w), min(n, i1 + w)
        cols = torch.cat([at[lo:hi], gl[(gl < lo) | (gl >= hi)]])
        S = torch.matmul(q[:, i0:i1], k[:, cols].transpose(1, 2)) / 8
        S.masked_fill_(~(((at[i0:i1, None] - cols[None, :]).abs() <= w) | glob[cols][None, :]), -math.inf)
        P = torch.softmax(S, dim=2)
        P = P * (~glob[i0:i1])[None, :, None]     # the global rows follow below
        O[:, i0:i1] = torch.matmul(P, v[:, cols])
        s[cols] += P.sum(dim=(0, 1))
    if gl.numel():
        P = torch.softmax(torch.matmul(q[:, gl], k.transpose(1, 2)) / 8, dim=2)
        O[:, gl] = torch.matmul(P, v)
        s += P.sum(dim=(0, 1))
    return O.transpose(0, 1), s / (H * n)


def _keep(case, s, alpha):
    """(kept mask, current indices of the tokens too near the threshold)."""
    n = s.numel()
    if case["rule"] == TOP_RATIO:
        kept = max(1, min(n, math.ceil(alpha * n)))
        order = torch.sort(s[1:], descending=True, stable=True)
        keep = torch.zeros(n, dtype=torch.bool, device=s.device)
        keep[0] = True
        keep[order.indices[: kept - 1] + 1] = True
        if kept - 1 in (0, n - 1):
            return keep, None
        theta = (order.values[kept - 2] + order.values[kept - 1]) / 2
    else:
        theta = alpha if case["rule"] == ABSOLUTE else alpha / n
        keep = s >= theta
        keep[0] = True
    near = (s - theta).abs() < MARGIN / n
    near[0] = False
    return keep, torch.nonzero(near)[:, 0]


def _alphas(case):
    nl = case["layers"]
    a = [case["a0"] + (case["a1"] - case["a0"]) * (l / (nl - 1) if nl > 1 else 0.0) for l in range(nl)]
    return torch.tensor(a, dtype=torch.float32).tolist()     # the values that the interface carries


def _walk(case, Q, K, V, pos, alphas, gpos, gen, scaled, out=None):
    """Runs the stack in 64 bits on Q, K, V [layers, B, L, H, 64] (rows by original position, redrawn in place where a
    score is too near its threshold), from the original positions ``pos`` of each sequence's first layer.  Returns
    the lengths [layer][sequence]; ``out``: where the results go."""
    dev, lens = Q.device, [[p.numel() for p in pos]]
    g = torch.tensor(gpos, device=dev)
    for l in range(case["layers"]):
        nxt = []
        for b, p in enumerate(pos):
            if not p.numel():
                nxt.append(p)
                continue
            gl = torch.nonzero(torch.isin(p, g))[:, 0]
            for _ in range(50):
                o, s = _attention(Q[l, b, p].double(), K[l, b, p].double(), V[l, b, p].double(), case["w"], gl)
                keep, near = _keep(case, s, alphas[l])
                if near is None or not near.numel():
                    break
                again = p[near]
                fresh = torch.randn((2, again.numel(), case["H"], HEAD), device=dev, generator=gen)
                Q[l, b, again] = fresh[0].to(Q.dtype)
                K[l, b, again] = (fresh[1] * scaled[b, again][:, None, None]).to(K.dtype)
            if out is not None:
                out["O"][l, b, : p.numel()], out["scores"][l, b, : p.numel()] = o, s
            nxt.append(p[keep])
        pos = nxt
        lens.append([p.numel() for p in pos])
    return lens


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _pruned(case):
    return case["rule"] != RELATIVE or case["a0"] > 0 or case["a1"] > 0


def _make(case, seed, out=None):
    """The case's inputs, and (``out`` given, or anything pruned) the walk through it in 64 bits."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    B, L, H, nl = case["B"], case["L"], case["H"], case["layers"]
    rand = lambda *shape: torch.rand(shape, device=dev, generator=gen)  # noqa: E731
    scaled = torch.ones((B, L), device=dev)
    count = int(round(case["frac"] * L))
    scaled.scatter_(1, rand(B, L).argsort(dim=1)[:, :count], case["scale"])
    gpos = [0] + sorted((1 + rand(L - 1).argsort()[: case["extra"]]).tolist())
    n0 = (L * (case["ragged"] + (1 - case["ragged"]) * rand(B))).long().clamp(1, L)
    n0[0] = L     # padded to the longest
    if case["kind"] == "encoder":
        return _make_encoder(case, gen, scaled, gpos, n0, out)
    Q, K, V = (torch.empty((nl, B, L, H, HEAD), dtype=torch.bfloat16, device=dev) for _ in range(3))
    for l in range(nl):
        Q[l] = torch.randn(Q.shape[1:], device=dev, generator=gen)
        K[l] = torch.randn(Q.shape[1:], device=dev, generator=gen) * scaled[:, :, None, None]
        V[l] = torch.randn(Q.shape[1:], device=dev, generator=gen)
    alphas = _alphas(case)
    rows = [torch.arange(int(n), device=dev) for n in n0]
    st = dict(Q=Q, K=K, V=V, n0=n0.int(), gpos=gpos, alphas=alphas)
    if case["kind"] == "layer":
        # tokens that survived earlier layers: token 0, and gaps between the positions of the others
        n0 = n0.clamp(max=max(1, int(0.9 * L)))
        st["n0"], rows = n0.int(), [torch.arange(int(n), device=dev) for n in n0]
        st["pos"] = torch.zeros((B, L), dtype=torch.int32, device=dev)
        for b in range(B):
            st["pos"][b, 1: int(n0[b])] = 1 + rand(L - 1).argsort()[: int(n0[b]) - 1].sort().values.int()
        # current indices stand for the positions in the walk: global where the position is
        current = [torch.nonzero(torch.isin(st["pos"][b, : int(n0[b])].long(), torch.tensor(gpos, device=dev)))[:, 0]
                   for b in range(B)]
        if _pruned(case) or out is not None:
            lens = [[int(n) for n in n0], []]
            for b in range(B):
                one = dict(case, B=1)
                sub = None if out is None else {k: out[k][:, b: b + 1] for k in out}
                r = _walk(one, Q[:, b: b + 1], K[:, b: b + 1], V[:, b: b + 1], [rows[b]], alphas,
                          current[b].tolist(), gen, scaled[b: b + 1], sub)
                lens[1] += r[1]
            st["lens"] = lens
    elif _pruned(case) or out is not None:
        st["lens"] = _walk(case, Q, K, V, rows, alphas, gpos, gen, scaled, out)
    st.setdefault("lens", [[int(n) for n in n0]] * (nl + 1))
    return st


def _norm(x, gamma, beta):
    return torch.nn.functional.layer_norm(x, (x.shape[-1],), gamma, beta, 1e-5)


def _make_encoder(case, gen, scaled, gpos, n0, out):
    """Hidden states of an encoder layer and random-init weights (no checkpoint is available).  The thresholds are
    absolute, one per sequence, as a calibrated model keeps them: each lies in the widest gap between neighbouring
    scores in the middle of its sequence's scores."""
    dev = scaled.device
    B, L, H = case["B"], case["L"], case["H"]
    D = H * HEAD
    randn = lambda *shape: torch.randn(shape, device=dev, generator=gen)  # noqa: E731
    mat = lambda o, i: (randn(o, i) / math.sqrt(i)).to(torch.bfloat16)  # noqa: E731
    X = randn(B, L, D).to(torch.bfloat16)
    W = dict(W_qkv=mat(3 * D, D), b_qkv=0.02 * randn(3 * D), W_o=mat(D, D), b_o=0.02 * randn(D),
             ln1_gamma=1 + 0.1 * randn(D), ln1_beta=0.1 * randn(D), W_1=mat(4 * D, D), b_1=0.02 * randn(4 * D),
             W_2=mat(D, 4 * D), b_2=0.02 * randn(D), ln2_gamma=1 + 0.1 * randn(D), ln2_beta=0.1 * randn(D))
    pos = torch.arange(L, device=dev).expand(B, L).contiguous().int()
    theta = torch.zeros(B, device=dev)
    W64 = {k: t.double() for k, t in W.items()}
    lens = [[int(n) for n in n0], []]
    for b in range(B):
        n = int(n0[b])
        x = X[b, :n].double()
        q, k, v = (x @ W64["W_qkv"].T + W64["b_qkv"]).view(n, 3, H, HEAD).unbind(1)
        o, s = _attention(q, k, v, case["w"], torch.tensor([g for g in gpos if g < n], device=dev))
        if n > 8:
            mid = torch.sort(s[1:]).values[int(0.35 * n): max(int(0.35 * n) + 2, int(0.65 * n))]
            gap = int((mid[1:] - mid[:-1]).argmax())
            theta[b] = (mid[gap] + mid[gap + 1]) / 2
        keep = s >= theta[b].double()
        keep[0] = True
        lens[1].append(int(keep.sum()))
        if out is not None:
            gelu = torch.nn.functional.gelu
            h1 = _norm(x[keep] + o.reshape(n, D)[keep] @ W64["W_o"].T + W64["b_o"], W64["ln1_gamma"], W64["ln1_beta"])
            f = gelu(h1 @ W64["W_1"].T + W64["b_1"])
            y = _norm(h1 + f @ W64["W_2"].T + W64["b_2"], W64["ln2_gamma"], W64["ln2_beta"])
            out["Y"][b, : y.shape[0]], out["O"][b, :n], out["scores"][b, :n] = y, o.reshape(n, D), s
    return dict(X=X, W=W, pos=pos, n0=n0.int(), gpos=gpos, theta=theta, lens=lens)


# ---------------------------------------------------------------------------
# what is measured
# ---------------------------------------------------------------------------
def prepare(case, seed):
    """Inputs, and what a program keeps between calls: the outputs (cleared: a call writes only the slots below each
    length) and the workspace."""
    st = _make(case, seed)
    dev = _device()
    B, L, H, nl = case["B"], case["L"], case["H"], case["layers"]
    zeros = lambda *shape, dtype=torch.float32: torch.zeros(shape, dtype=dtype, device=dev)  # noqa: E731
    st["case"] = case
    if case["kind"] == "encoder":
        st["out"] = {"Y": zeros(B, L, H * HEAD, dtype=torch.bfloat16), "O": zeros(B, L, H * HEAD, dtype=torch.bfloat16),
                     "scores": zeros(B, L), "pos_out": zeros(B, L, dtype=torch.int32), "len_out": zeros(B, dtype=torch.int32)}
        st["ws"] = sc.new_encoder_workspace(B, L, H, dev)
        return st
    if case["kind"] == "layer":
        st["out"] = {"O": zeros(B, L, H, HEAD, dtype=torch.bfloat16), "scores": zeros(B, L),
                     "pos_out": zeros(B, L, dtype=torch.int32), "len_out": zeros(B, dtype=torch.int32)}
        st["Q"], st["K"], st["V"] = st["Q"][0], st["K"][0], st["V"][0]
        st["ws"] = sc.new_workspace(B, L, H, dev)
        return st
    st["mask"] = None
    if case["ragged"] < 1:
        st["mask"] = (torch.arange(L, device=dev)[None, :] < st["n0"][:, None]).to(torch.uint8)
    if case["kind"] == "host":
        for k in ("Q", "K", "V", "mask"):
            if st[k] is not None:
                st[k] = torch.empty(st[k].shape, dtype=st[k].dtype, pin_memory=True).copy_(st[k])
        st["out"] = sc.new_host_outputs(nl, B, L, H)
        for t in st["out"].values():
            t.zero_()
        st["ws"] = sc.new_stack_host_workspace(nl, B, L, H, dev)
        return st
    st["out"] = {"O": zeros(nl, B, L, H, HEAD, dtype=torch.bfloat16), "scores": zeros(nl, B, L),
                 "pos": zeros(nl + 1, B, L, dtype=torch.int32), "len": zeros(nl + 1, B, dtype=torch.int32)}
    st["ws"] = sc.new_workspace(B, L, H, dev)
    return st


def run(st):
    c = st["case"]
    if c["kind"] == "encoder":
        return sc.encoder_layer_forward(st["X"], st["n0"], st["pos"], c["w"], st["gpos"], st["W"], theta=st["theta"],
                                        out=st["out"], workspace=st["ws"])
    if c["kind"] == "layer":
        sc.layer_forward(st["Q"], st["K"], st["V"], st["n0"], st["pos"], c["w"], st["gpos"], st["alphas"][0],
                         keep_rule=c["rule"], workspace=st["ws"], **st["out"])
        return st["out"]
    call = sc.stack_forward_host if c["kind"] == "host" else sc.stack_forward
    return call(st["Q"], st["K"], st["V"], st["mask"], st["gpos"], c["w"], st["alphas"], out=st["out"],
                workspace=st["ws"], keep_rule=c["rule"])


def exact(case, seed):
    """The floating outputs of ``run`` in 64 bits (None in the place of the whole-valued ones), zero where the call
    writes nothing."""
    dev = _device()
    B, L, H, nl = case["B"], case["L"], case["H"], case["layers"]
    zeros = lambda *shape: torch.zeros(shape, dtype=torch.float64, device=dev)  # noqa: E731
    if case["kind"] == "encoder":
        out = {"Y": zeros(B, L, H * HEAD), "O": zeros(B, L, H * HEAD), "scores": zeros(B, L)}
        _make(case, seed, out)
        return dict(out, pos_out=None, len_out=None)
    out = {"O": zeros(nl, B, L, H, HEAD), "scores": zeros(nl, B, L)}
    _make(case, seed, out)
    if case["kind"] == "layer":
        return {"O": out["O"][0], "scores": out["scores"][0], "pos_out": None, "len_out": None}
    return dict(out, pos=None, len=None)


@functools.lru_cache(maxsize=64)
def _lengths(items):
    return _make(dict(items), 1)["lens"]


def _pairs(n, w, globals_):
    """Allowed (query, key) pairs of one sequence: the band, and the global rows and columns outside it."""
    m = min(w, n - 1)
    band = n * (2 * m + 1) - m * (m + 1)
    return min(n * n, band + 2 * min(globals_, n) * max(0, n - 2 * m - 1))


def work(case):
    """Per layer and sequence of n tokens: Q, K, V read, O, the score and the position written, once each; 4 * 64 flops
    per head and allowed pair (Q K^T and P V).  An encoder layer: its products, its weights once, X in and Y out.
    The lengths after pruning are those of the inputs of seed 1."""
    B, H, w = case["B"], case["H"], case["w"]
    D = H * HEAD
    lens = _lengths(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    nbytes = flops = 0.0
    for l in range(case["layers"]):
        for b in range(B):
            n = lens[l][b]
            if not n:
                continue
            flops += 4 * HEAD * H * _pairs(n, w, 1 + case["extra"])
            if case["kind"] == "encoder":
                kept = lens[1][b]
                flops += 2 * n * D * 3 * D + 2 * kept * D * (D + 8 * D)
                nbytes += n * (2 * D + 2 * D + 8) + kept * 2 * D
            else:
                nbytes += n * (8 * D + 8)
    if case["kind"] == "encoder":
        nbytes += 2 * 12 * D * D + 4 * 13 * D
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """O (and Y) are bf16 of probabilities rounded to bf16: 2e-3 off the 64-bit values in the 2-norm, so two correct
    implementations may lie 3e-3 apart.  Kept lists are whole numbers, clear of their thresholds."""
    return {"rel": 1e-2, "max": 0.3}

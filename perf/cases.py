"""The work that programs built on this library have it do, as cases that can be timed.

Each case is one pass through the public entry points of
``paper_2607_08991_gb300.sats`` at sizes a user runs: decode of one token and of
batches, prefill, whole decoder stacks with and without token routing, the
LoRA-aware path, and the calibrations that a deployment runs once per model.
Weights are synthetic bf16 ~ N(0, 0.02) and activations ~ N(0, 1), as in this
repository's workloads.

Thresholds are percentiles of the post-gate magnitudes of the case's own tokens,
moved to the middle of the widest gap between neighbouring magnitudes near that
percentile: two correct implementations then keep the same neurons, and outputs
can be compared closely although the mask itself is a step function.
"""
import math

import numpy as np
import torch

from paper_2607_08991_gb300 import sats

LLAMA = dict(H=4096, N=14336)
QWEN = dict(H=4096, N=12288)
STD = 0.02


# ---------------------------------------------------------------------- the cases
def listed():
    return [
        # decode of one token on a layer of a few MB (on-device draft models): latency only
        dict(name="small_decode_1", kind="layer", H=512, N=1408, B=1, x="bf16", s=0.5, lists=True),
        # decode of one token, the library's main use, kept lists for the caller's own bookkeeping
        dict(name="llama_decode_1", kind="layer", B=1, x="bf16", s=0.7, lists=True, **LLAMA),
        # batched decode, a few concurrent requests
        dict(name="llama_decode_8", kind="layer", B=8, x="bf16", s=0.5, lists=True, **LLAMA),
        # batched decode of a busy server, a ragged batch of fp32 activations
        dict(name="llama_decode_101_f32", kind="layer", B=101, x="f32", s=0.8, lists=False, **LLAMA),
        # prefill of a long prompt
        dict(name="llama_prefill_2048", kind="layer", B=2048, x="bf16", s=0.6, lists=False, **LLAMA),
        # one decode step of a whole unrouted model
        dict(name="llama_stack_decode_1", kind="stack", L=32, B=1, s=0.7, eps=1e-5, V=0, dense=0.0, **LLAMA),
        # one decode step of a whole routed model for a batch of requests
        dict(name="qwen_stack_routed_8", kind="stack", L=36, B=8, s=0.5, eps=1e-6, V=151936, dense=0.3, **QWEN),
        # routed prefill of a short, ragged prompt through one block
        dict(name="llama_block_routed_333", kind="stack", L=1, B=333, s=0.6, eps=1e-5, V=128256, dense=0.2, **LLAMA),
        # decode of a few requests on a fine-tuned model (LoRA adapters folded into the sparse path)
        dict(name="llama_lora_decode_4", kind="lora", B=4, r=16, x="bf16", s=0.7, **LLAMA),
        # percentile (CATS) threshold of a layer from calibration vectors
        dict(name="llama_threshold_256", kind="threshold", B=256, x="bf16", s=0.7, **LLAMA),
        # sensitivity-aware (SATS) thresholds of consecutive blocks; a model runs this over all its blocks
        dict(name="llama_calibrate_2x64", kind="calibrate", L=2, C=64, K0=20, K1=8, s=0.5, eps=1e-5, **LLAMA),
        # routing table of a vocabulary from corpus losses, then the routing of a prompt with it
        dict(name="routing_table_1m", kind="routing", V=151936, n=1000000, m=250000, s=0.5, B=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _layer_size(rng):
    """Hidden sizes in multiples of 8, any number of neurons; at most the Llama-shaped layer's weights."""
    H = 8 * _log(rng, 32, 1024)
    N = min(_log(rng, 1.5 * H, 5 * H) | rng.randint(0, 1), LLAMA["H"] * LLAMA["N"] // H)
    return H, N


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "stack", "stack", "lora", "threshold", "calibrate", "routing"])
    H, N = _layer_size(rng)
    s = round(rng.uniform(0.4, 0.92), 3)
    if kind == "layer":
        B = _log(rng, 1, 2048)
        # s = 0 is the base (dense) layer
        return dict(kind=kind, H=H, N=N, B=B, x=rng.choice(["bf16", "f32"]), s=rng.choice([0.0, s, s, s]),
                    lists=rng.random() < 0.4)
    if kind == "stack":
        routed = rng.random() < 0.7
        # (deep stacks at small batches only: a mask decision that rounding turns in one block of a large
        # batch turns many more in the blocks after it, and two correct results can no longer be compared)
        B = _log(rng, 1, 1024)
        return dict(kind=kind, H=H, N=N, L=_log(rng, 1, 32 if B <= 2 else 4 if B <= 8 else 1), B=B, s=s, eps=1e-6,
                    V=_log(rng, 1000, 160000) if routed else 0, dense=round(rng.uniform(0.1, 0.5), 2) if routed else 0.0)
    if kind == "lora":
        return dict(kind=kind, H=H, N=N, B=_log(rng, 1, 16), r=rng.choice([8, 16, 24, 32]),
                    x=rng.choice(["bf16", "f32"]), s=s)
    if kind == "threshold":
        return dict(kind=kind, H=H, N=N, B=_log(rng, 16, 512), x=rng.choice(["bf16", "f32"]), s=s)
    if kind == "calibrate":
        return dict(kind=kind, H=H, N=N, L=2, C=_log(rng, 8, 64), K0=rng.randint(8, 20),
                    K1=rng.randint(3, 8), s=round(rng.uniform(0.3, 0.7), 2), eps=1e-6)
    return dict(kind=kind, V=_log(rng, 2000, 160000), n=_log(rng, 50000, 1000000), m=_log(rng, 10000, 250000),
                s=round(rng.uniform(0.2, 0.8), 2), B=_log(rng, 16, 4096))


# ---------------------------------------------------------------------- inputs
def _gen(seed, *tags):
    g = torch.Generator(device="cuda")
    v = int(seed) & 0x7FFFFFFF
    for t in tags:
        v = (v * 1000003 + int(t) + 17) & 0x7FFFFFFFFFFF
    g.manual_seed(v)
    return g


def _normal(shape, seed, *tags, std=1.0, dtype=torch.float32):
    return torch.randn(shape, generator=_gen(seed, *tags), device="cuda").mul_(std).to(dtype)


def _weights(case, seed, layer):
    """W_gate, W_up [H][N] and W_down [N][H] of one block."""
    H, N = case["H"], case["N"]
    return tuple(_normal(shape, seed, 1, layer, k, std=STD, dtype=torch.bfloat16)
                 for k, shape in enumerate(((H, N), (H, N), (N, H))))


def _layer(case, seed, layer=0):
    w = _weights(case, seed, layer)
    return sats.Layer(*w), w


def _x(case, seed):
    B = case.get("B", case.get("C"))
    return _normal((B, case["H"]), seed, 2, dtype=torch.bfloat16 if case.get("x") == "bf16" else torch.float32)


def _norm_w(case, seed, layer):
    return 1.0 + _normal((case["H"],), seed, 3, layer, std=0.02)


def _adapter(case, seed):
    """A_gate [H][r], B_gate [r][N], A_up, B_up, A_down [N][r], B_down [r][H]."""
    H, N, r = case["H"], case["N"], case["r"]
    shapes = ((H, r), (r, N), (H, r), (r, N), (N, r), (r, H))
    return [_normal(shape, seed, 4, k, std=STD, dtype=torch.bfloat16) for k, shape in enumerate(shapes)]


def _silu(g):
    return g / (1.0 + torch.exp(-g))


def _gap_threshold(a, s):
    """The s-quantile of |a|, moved to the middle of the widest gap within 1 % of the values around it."""
    if s <= 0.0 or a.numel() == 0:
        return 0.0
    v = a.abs().flatten().sort().values
    n = v.numel()
    w = max(4, int(0.01 * n))
    i0 = min(max(0, int(s * n) - w), max(0, n - 2))
    i1 = min(n - 1, i0 + 2 * w)
    if i1 <= i0:
        return float(v[i0])
    gap = v[i0 + 1:i1 + 1] - v[i0:i1]
    k = i0 + int(gap.argmax())
    return float(np.float32(0.5 * (float(v[k]) + float(v[k + 1]))))


def _rms(x, w, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * w


def _ids(case, seed, n, V, tag):
    """Zipf(1.1) token ids over the vocabulary, through the explicit CDF."""
    cdf = torch.arange(1, V + 1, device="cuda", dtype=torch.float64).pow(-1.1).cumsum(0)
    u = torch.rand(n, generator=_gen(seed, 5, tag), device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u, right=True).clamp_(max=V - 1).to(torch.int32)


def _routing(case, seed):
    """Token ids and the table of a routed stack (1 = base path)."""
    V = case["V"]
    if not V:
        return None, None
    lut = (torch.rand(V, generator=_gen(seed, 6), device="cuda") < case["dense"]).to(torch.uint8)
    return _ids(case, seed, case["B"], V, 0), lut


def _mlp(n, w, t, dtype, lora=None, last=False):
    """The thresholded gated MLP of rows n at per-row thresholds t [B][1] in plain torch; with `last`
    only the post-gate activations."""
    Wg, Wu, Wd = w
    g = n @ Wg.to(dtype)
    if lora is not None:
        Ag, Bg, Au, Bu, Ad, Bd = (m.to(dtype) for m in lora)
        g = g + (n @ Ag) @ Bg
    a = _silu(g)
    if last:
        return a
    u = n @ Wu.to(dtype)
    if lora is not None:
        u = u + (n @ Au) @ Bu
    h = torch.where(a.abs() >= t, a, torch.zeros_like(a)) * u
    y = h @ Wd.to(dtype)
    if lora is not None:
        y = y + (h @ Ad) @ Bd
    return y


def _corpus(case, seed):
    """Corpus occurrences with the two paths' losses, and a held-out split."""
    V, n = case["V"], case["n"]
    ids = _ids(case, seed, n, V, 1)
    risk = torch.empty(V, device="cuda").exponential_(10.0, generator=_gen(seed, 7))
    l_base = 3.0 + _normal((n,), seed, 8)
    l_sparse = l_base + risk[ids.long()] + _normal((n,), seed, 9, std=0.05)
    return ids, l_base, l_sparse, _ids(case, seed, case["m"], V, 2)


# ---------------------------------------------------------------------- what a program has in hand
class _State:
    pass


def prepare(case, seed):
    S = _State()
    S.case = case
    kind = case["kind"]
    if kind == "routing":
        S.ids, S.l_base, S.l_sparse, S.held = _corpus(case, seed)
        S.prompt = _ids(case, seed, case["B"], case["V"], 3)
        S.perm = torch.zeros(case["B"], dtype=torch.int32, device="cuda")
        S.n_dense = torch.zeros(1, dtype=torch.int32, device="cuda")
        return S
    H, N = case["H"], case["N"]
    if kind in ("layer", "lora"):
        B = case["B"]
        S.layer, w = _layer(case, seed)
        S.x = _x(case, seed)
        lora = None
        if kind == "lora":
            lora = _adapter(case, seed)
            S.lora = sats.Lora(S.layer, *lora, scale=1.0)
        S.t = 0.0
        if case["s"] > 0.0:
            S.t = _gap_threshold(_mlp(S.x.float(), w, None, torch.float32, lora, last=True), case["s"])
        S.ws = sats.Workspace(H, N, B)
        S.y = torch.zeros((B, H), device="cuda")
        S.idx = S.cnt = None
        if case.get("lists"):
            S.idx = torch.full((B, N), -1, dtype=torch.int32, device="cuda")
            S.cnt = torch.zeros(B, dtype=torch.int32, device="cuda")
        return S
    if kind == "stack":
        B, L = case["B"], case["L"]
        S.ids, S.lut = _routing(case, seed)
        S.x_in = _x(case, seed)
        S.x = S.x_in.clone()
        S.ws = sats.Workspace(H, N, B)
        S.layers, S.norm_w, S.t = [], [], []
        base = None if S.ids is None else (S.lut[S.ids.long()] != 0).unsqueeze(1)
        x = S.x_in
        for l in range(L):
            layer, w = _layer(case, seed, l)
            S.layers.append(layer)
            S.norm_w.append(_norm_w(case, seed, l))
            n = _rms(x, S.norm_w[l], case["eps"])
            a = _mlp(n, w, None, torch.float32, last=True)
            t = _gap_threshold(a if base is None else a[~base.squeeze(1)], case["s"])
            S.t.append(t)
            if l + 1 < L:
                tt = torch.full((B, 1), t, device="cuda")
                x = x + _mlp(n, w, tt if base is None else torch.where(base, torch.zeros_like(tt), tt), torch.float32)
        return S
    if kind == "threshold":
        S.layer, _ = _layer(case, seed)
        S.x = _x(case, seed)
        S.a = torch.zeros((case["B"], N), device="cuda")
        S.sel = torch.zeros(sats.select_workspace_bytes(), dtype=torch.uint8, device="cuda")
        return S
    # calibrate
    S.layers = [_layer(case, seed, l)[0] for l in range(case["L"])]
    S.norm_w = [_norm_w(case, seed, l) for l in range(case["L"])]
    S.x = _x(case, seed)
    return S


# ---------------------------------------------------------------------- one pass
def run(S):
    case = S.case
    kind = case["kind"]
    if kind == "layer":
        if case["s"] <= 0.0 and case["x"] == "bf16" and S.idx is None:
            sats.dense_mlp(S.layer, S.x, S.y, S.ws)
        elif case["x"] == "bf16":
            sats.sparse_mlp(S.layer, S.x, S.t, S.y, S.ws, S.idx, S.cnt)
        else:
            sats.sparse_mlp_f32(S.layer, S.x, S.t, S.y, S.ws, S.idx, S.cnt)
        # (entries of a row of idx past its count are unspecified; here they keep what prepare() wrote)
        return dict(y=S.y) if S.idx is None else dict(y=S.y, idx=S.idx, cnt=S.cnt)
    if kind == "lora":
        sats.sparse_mlp_lora(S.layer, S.lora, S.x, S.t, S.y, S.ws)
        return dict(y=S.y)
    if kind == "stack":
        S.x.copy_(S.x_in)   # the residual stream starts as this step's embeddings
        sats.mlp_stack(S.layers, S.norm_w, S.t, case["eps"], S.x, S.ws, token_ids=S.ids, lut=S.lut)
        return dict(x=S.x)
    if kind == "threshold":
        if case["x"] == "bf16":
            sats.gate_act(S.layer, S.x, S.a)
        else:
            sats.gate_act_f32(S.layer, S.x, S.a)
        return dict(a=S.a, t=float(sats.percentile_threshold(S.a, case["s"], S.sel)))
    if kind == "calibrate":
        r = sats.sats_calibrate(S.layers, S.norm_w, case["eps"], S.x, case["s"], K0=case["K0"], K1=case["K1"])
        t, err, sp = (np.asarray(v, dtype=np.float64) for v in r["table"])
        return dict(t=np.asarray(r["t"], dtype=np.float64), b=float(r["b"]), S=float(r["S"]), table_t=t, table_err=err,
                    table_sp=sp)
    score = sats.token_scores(S.ids, S.l_base, S.l_sparse, case["V"])
    tau, R, lut = sats.route_calibrate(score, S.held, case["s"])
    sats.route(S.prompt, lut, S.perm, S.n_dense)
    return dict(score=score, tau=float(tau), R=float(R), lut=lut, perm=S.perm, n_dense=S.n_dense)


# ---------------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "routing":
        return dict(bytes=12 * case["n"] + 4 * case["m"] + 5 * case["V"] + 9 * case["B"], flops=2 * case["n"])
    H, N = case["H"], case["N"]
    xb = 2 if case.get("x") == "bf16" else 4
    if kind in ("layer", "lora"):
        B, s = case["B"], case["s"]
        # all of W_gate, the W_up columns and W_down rows that some token keeps
        bytes_ = 2 * H * N + 4 * H * N * (1.0 - s ** B) + B * H * (xb + 4)
        flops = B * H * N * (2 + 4 * (1.0 - s))
        if case.get("lists"):
            bytes_ += 4 * B * (N * (1.0 - s) + 1)
        if kind == "lora":
            r = case["r"]
            bytes_ += 6 * r * (H + N)
            flops += 6 * B * r * (H + N)
        return dict(bytes=bytes_, flops=flops)
    if kind == "stack":
        B, s, d = case["B"], case["s"], case["dense"] if case["V"] else 0.0
        kept = d + (1.0 - d) * (1.0 - s)
        return dict(bytes=case["L"] * (2 * H * N + 4 * H * N * (1.0 - (1.0 - kept) ** B)) + 8 * B * H,
                    flops=case["L"] * B * H * N * (2 + 4 * kept))
    if kind == "threshold":
        B = case["B"]
        return dict(bytes=2 * H * N + B * H * xb + 4 * B * N, flops=2 * B * H * N)
    # calibrate: gate, up and the dense output of every block, and the candidates' dropped neurons
    # once per pass over the candidates (each neuron falls between two neighbouring thresholds)
    C, L = case["C"], case["L"]
    return dict(bytes=L * 6 * H * N + 4 * C * H, flops=L * C * H * N * (6 + 2 * 2))


def tolerance(case):
    """About four times the largest error against exact() that was measured over the listed and drawn cases."""
    kind = case["kind"]
    if kind == "routing":
        return dict(rel=1e-6, max=1e-5, differ=1e-5)
    if kind == "threshold":
        return dict(rel=2e-6, max=2e-5)
    if kind == "calibrate":
        # shares of C * N neurons and errors of single candidates: one neuron at a threshold counts
        return dict(rel=1e-3, max=1e-2)
    if case["B"] <= 2 or kind == "lora":
        return dict(rel=1e-5, max=1e-4, differ=0.01) if kind != "stack" else dict(rel=5e-5, max=5e-4)
    # batches on the tensor cores: 1.2e-5 without a turned mask decision; with B * N magnitudes around one
    # threshold some decisions turn (5e-4 at 2048 tokens), each a neuron's share of one token's output
    if case["s"] <= 0.0:
        return dict(rel=5e-5, max=5e-4)
    # (a deep stack carries each turned decision on: two passes on the same inputs are up to 6e-3 apart)
    return dict(rel=2e-3 if case.get("L", 1) == 1 else 0.03, max=0.2, differ=0.01)


# ---------------------------------------------------------------------- the same in 64 bits, in plain torch
def exact(case, seed):
    kind = case["kind"]
    D = torch.float64
    if kind == "routing":
        return _exact_routing(case, seed)
    if kind == "calibrate":
        return _exact_calibrate(case, seed)
    if kind == "threshold":
        a = _mlp(_x(case, seed).to(D), _weights(case, seed, 0), None, D, last=True)
        v = a.abs().flatten().sort().values
        m = max(1, math.ceil(case["s"] * v.numel() * (1.0 - 2.0 ** -50)))
        return dict(a=a, t=float(v[m - 1]))
    if case.get("L", 1) > 1 and case["B"] > 2:
        return None   # blocks after a turned mask decision work on another input: no one value to be near to
    S = prepare(case, seed)   # for its thresholds
    if kind in ("layer", "lora"):
        lora = _adapter(case, seed) if kind == "lora" else None
        y = _mlp(S.x.to(D), _weights(case, seed, 0), torch.full((case["B"], 1), S.t, device="cuda", dtype=D), D, lora)
        return dict(y=y) if S.idx is None else dict(y=y, idx=None, cnt=None)
    x = S.x_in.to(D)
    base = None if S.ids is None else (S.lut[S.ids.long()] != 0).unsqueeze(1)
    for l in range(case["L"]):
        t = torch.full((case["B"], 1), S.t[l], device="cuda", dtype=D)
        if base is not None:
            t = torch.where(base, torch.zeros_like(t), t)
        x = x + _mlp(_rms(x, S.norm_w[l].to(D), case["eps"]), _weights(case, seed, l), t, D)
    return dict(x=x)


def _exact_routing(case, seed):
    """Per-token mean excess loss, the held-out share below each candidate tau, and the nearest to the target."""
    ids, l_base, l_sparse, held = _corpus(case, seed)
    V = case["V"]
    d = (l_sparse - l_base).clamp(min=0.0).double()   # the excess loss itself is a 32-bit difference
    total = torch.zeros(V, device="cuda", dtype=torch.float64).index_add_(0, ids.long(), d)
    count = torch.bincount(ids.long(), minlength=V)
    score = torch.where(count > 0, total / count, torch.full_like(total, math.inf))
    sc = score[held.long()].cpu().numpy()
    cand = np.unique(np.concatenate([[0.0], sc, [np.inf]]))
    R = np.searchsorted(np.sort(sc), cand, side="left") / case["m"]
    k = int(np.argmin(np.abs(R - case["s"])))
    return dict(score=score, tau=float(cand[k]), R=float(R[k]), lut=None, perm=None, n_dense=None)


def _select(t, err, sp, target, guard, guard_t, guard_sp):
    """The budget whose thresholds come nearest to the target sparsity; per block the largest threshold within it."""
    L = t.shape[0]
    best = None
    for b in np.unique(np.concatenate([[0.0], err.ravel()])):
        pick, share = [], 0.0
        for l in range(L):
            if l == guard:
                pick.append(guard_t)
                share += guard_sp
                continue
            ok = (err[l] <= b) & (t[l] > 0.0)
            k = int(np.argmax(np.where(ok, t[l], -1.0))) if ok.any() else -1
            pick.append(float(t[l][k]) if k >= 0 else 0.0)
            share += float(sp[l][k]) if k >= 0 else 0.0
        gap = abs(share / L - target)
        if best is None or gap < best[0]:
            best = (gap, float(b), pick, share / L)
    return best[1:]


def _exact_calibrate(case, seed):
    D = torch.float64
    L, C, K0, K1, N = case["L"], case["C"], case["K0"], case["K1"], case["N"]
    x = _x(case, seed).to(D)
    blocks, tc, top = [], [], []
    guard_t = 0.0
    for l in range(L):
        w = _weights(case, seed, l)
        n = _rms(x, _norm_w(case, seed, l).to(D), case["eps"])
        a = _mlp(n, w, None, D, last=True)
        h = a * (n @ w[1].to(D))
        y = h @ w[2].to(D)
        v = a.abs().flatten().sort().values
        rank = lambda k: float(v[max(1, math.ceil(k * v.numel() * (1.0 - 2.0 ** -50))) - 1])  # noqa: E731
        tc.append([rank(k / K0) for k in range(1, K0)])
        top.append(float(v[-1]))
        if l == L - 1:
            guard_t = rank(case["s"])
        blocks.append((w, a.abs(), h, y))
        x = x + y
    tc = np.asarray(tc)

    def errors(l, ts):
        w, a, h, y = blocks[l]
        wd = w[2].to(D)
        e, p = [], []
        for t in ts:
            drop = a < t
            e.append(float((torch.where(drop, h, torch.zeros_like(h)) @ wd).norm(dim=1).div(y.norm(dim=1) + 1e-6).mean()))
            p.append(float(drop.double().mean()))
        return e, p

    ec, sc = (np.asarray(v) for v in zip(*(errors(l, tc[l]) for l in range(L))))
    guard_sp = errors(L - 1, [guard_t])[1][0]
    _, t0, _ = _select(tc, ec, sc, case["s"], L - 1, guard_t, guard_sp)
    rows = []
    for l in range(L):
        below, above = tc[l][tc[l] < t0[l]], tc[l][tc[l] > t0[l]]
        lo = float(below.max()) if below.size else 0.0
        hi = float(above.min()) if above.size else top[l]
        tf = [lo + (hi - lo) * (k + 1) / (K1 + 1) for k in range(K1)]
        ef, sf = errors(l, tf)
        rows.append((np.concatenate([tc[l], tf]), np.concatenate([ec[l], ef]), np.concatenate([sc[l], sf])))
    ta, ea, sa = (np.stack(v) for v in zip(*rows))
    b, t, S = _select(ta, ea, sa, case["s"], L - 1, guard_t, guard_sp)
    return dict(t=np.asarray(t), b=b, S=S, table_t=ta, table_err=ea, table_sp=sa)

"""The calls this library is used for, as measurable cases.

A case is one call (or the few calls) a program makes through the public
binding ``paper_2603_00188_gb300.stlite``: the whole compression pass on one
layer, on all layers of a model and on a packed batch; its staged entry points
(the score, gate and saliency maps; selection and compaction); attention over
the cache while decoding; and the prompt-wide base score.  Sizes are those of
the repository's workloads (``synth.py``), the ranges of ``draw`` are around
them.  Keys follow the same recipe as there: screenshot frames that drift from
step to step or repeat, planted UI boxes the window attends to, and text.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2603_00188_gb300 import stlite

D = 128
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------- cases

def _compress(name, **kw):
    c = dict(name=name, kind="compress", dtype="bf16", layers=1, seqs=1, frames=10, gh=36, gw=64, text=64,
             ragged=0, hq=28, hkv=4, w=32, beta=0.2, css=3, tsg=1, heavy=False, exact_dups=False)
    c.update(kw)
    return c


def listed():
    return [
        # the fp32 reference layer a user checks an integration with: the smallest whole pass, latency-bound
        _compress("layer_fp32_tiny", dtype="f32", frames=4, gh=16, gw=16, text=32),
        # one layer of a 10-screenshot session at the largest patch grid, compressed as its prefill finishes
        _compress("layer_uitars"),
        # every layer of a 50-step session at once (the library's headline workload, the largest call)
        _compress("layers_traj50", layers=28, frames=50, gh=32, gw=32, text=48),
        # a batch of sessions of different lengths, every layer, smaller backbone, hard budget
        _compress("varlen_small_backbone", layers=28, seqs=8, frames=20, ragged=8, gh=24, gw=42, text=40, hq=12,
                  hkv=2, w=16, beta=0.1),
        # one layer of a 100-step session: ragged row tiles, 448 query rows per KV head, exact duplicate frames
        _compress("layer_long_horizon", frames=100, gh=36, gw=36, text=32, w=64, beta=0.1, heavy=True,
                  exact_dups=True),
        # the second step of a session, every layer: small launches, as at the start of each trajectory
        _compress("layers_second_step", layers=28, frames=2, gh=32, gw=32, text=48),
        # score, gate and saliency maps of an fp32 layer (a policy of the user's own combines them)
        dict(_compress("maps_fp32", dtype="f32", frames=5), kind="maps"),
        # the same maps of a bf16 layer whose screenshots differ in size, odd grids among them
        dict(_compress("maps_ragged", frames=14, gh=35, gw=61, text=37, ragged=2), kind="maps"),
        # Top-B and compaction of one long layer from maps the program already has
        dict(_compress("pick_traj50", frames=50, gh=32, gw=32, text=48), kind="pick"),
        # one decoding step over every layer's compressed cache
        dict(name="decode_layers", kind="decode", dtype="bf16", layers=28, n=10720, hq=28, hkv=4, w=1),
        # one layer of a decoding step (layers run one after another in a model), tokens appended since
        dict(name="decode_one_layer", kind="decode", dtype="bf16", layers=1, n=10757, hq=28, hkv=4, w=1),
        # the Mean Attention base over the whole prompt of an 8-step session
        dict(name="prompt_mean", kind="prompt", dtype="bf16", n=8576, rows=8576, hq=28, hkv=4, mean=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


HEADS = [(28, 4), (12, 2), (14, 2), (16, 8), (32, 8), (40, 8)]


def draw(rng):
    """One more case of the same ranges (odd grids, head counts, windows,
    budgets and lengths), at most the cost of the largest listed one."""
    kind = rng.choice(["compress", "compress", "compress", "varlen", "maps", "maps", "pick", "decode", "prompt"])
    hq, hkv = rng.choice(HEADS)
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    if kind == "decode":
        return dict(kind="decode", dtype=dtype, layers=rng.choice([1, 1, 24, 28]), n=_log(rng, 60, 30000 if dtype == "bf16" else 8000),
                    hq=hq, hkv=hkv, w=rng.choice([1, 1, 1, 4]))
    if kind == "prompt":
        n = _log(rng, 300, 8500 if dtype == "bf16" else 1200)
        return dict(kind="prompt", dtype=dtype, n=n, rows=rng.choice([n, max(1, n // 3), max(1, n - 77)]), hq=hq,
                    hkv=hkv, mean=rng.random() < 0.5)
    while True:
        c = _compress("", dtype=dtype, frames=_log(rng, 1, 60), gh=rng.randint(9, 44), gw=rng.randint(9, 76),
                      text=rng.randint(0, 70), ragged=rng.choice([0, 0, 0, 2]), hq=hq, hkv=hkv,
                      w=rng.choice([1, 8, 16, 31, 32, 32, 64]), beta=rng.choice([0.05, 0.1, 0.2, 0.2, 0.3, 0.4]),
                      css=rng.choice([3, 3, 3, 3, 5]), tsg=rng.choice([1, 1, 1, 1, 0]), heavy=rng.random() < 0.2,
                      exact_dups=rng.random() < 0.3)
        del c["name"]
        c["kind"] = "compress" if kind == "varlen" else kind
        if kind == "varlen":
            c.update(seqs=rng.randint(2, 8), ragged=min(4, c["frames"] - 1), frames=max(2, c["frames"] // 2))
        if kind in ("compress", "varlen"):
            c["layers"] = rng.choice([1, 1, 4, 24, 28])
        f = work(c)["flops"]
        if f <= (1.2e12 if dtype == "bf16" else 1.5e10) and c["layers"] * sum(_tokens(c)) <= 1_400_000:
            return c


# ------------------------------------------------------------------ layout

def _layouts(case):
    """One (offset, grid_h, grid_w) per sequence.  ragged: for one sequence,
    every ragged-th frame is a smaller screenshot; for a batch, each sequence
    has up to that many frames fewer than the longest."""
    out = []
    for s in range(case["seqs"]):
        r = random.Random(1000 * s + case["frames"])
        frames = case["frames"]
        if case["seqs"] > 1 and s:
            frames = max(1, frames - r.randint(0, case["ragged"]))
        off, gh, gw, at = [], [], [], 0
        for f in range(frames):
            a, b = case["gh"], case["gw"]
            if case["seqs"] == 1 and case["ragged"] and f % case["ragged"]:
                a, b = max(1, a - r.randint(1, a // 2)), max(1, b - r.randint(1, b // 2))
            off.append(at)
            gh.append(a)
            gw.append(b)
            at += a * b + case["text"]
        out.append((tuple(np.array(x, np.int32) for x in (off, gh, gw)), at))
    return out


def _tokens(case):
    return [n for _, n in _layouts(case)]


# ------------------------------------------------------------------ inputs

def _normal(gen, shape, heavy=False):
    z = torch.randn(shape, generator=gen, device="cuda")
    if heavy:  # Student-t, three degrees of freedom
        z /= (torch.randn((3, *shape), generator=gen, device="cuda").square_().sum(0) / 3).sqrt_()
    return z


def _keys(case, frames, n, q, gen, rnd):
    """Keys [L][n][Hkv][d] of one sequence of every layer (see the module's docstring)."""
    L, hkv, heavy = case["layers"], case["hkv"], case["heavy"]
    k = torch.empty((L, n, hkv, D), dtype=DTYPES[case["dtype"]], device="cuda")
    qhat = q.float().view(L, case["w"], hkv, -1, D).mean((1, 3))
    qhat = qhat / qhat.norm(dim=-1, keepdim=True)
    bg = prev = None
    copies = 0
    for f, (off, gh, gw) in enumerate(zip(*(x.tolist() for x in frames))):
        size = gh * gw
        same = prev is not None and prev.shape[1] == size
        if same and copies > 0:
            copies -= 1
            frame = prev
        elif same and not case["exact_dups"] and rnd.random() < 0.3:  # a near-duplicate screenshot
            frame = prev + 0.01 * _normal(gen, prev.shape)
        else:
            if bg is None or bg.shape[1] != size:
                bg = _normal(gen, (L, size, hkv, D), heavy)
            else:
                bg = bg + 0.1 * _normal(gen, bg.shape)
            frame = bg.clone()
            cells = set()
            for _ in range(rnd.randint(5, 20)):
                bh, bw = (1, 2) if case["exact_dups"] else (rnd.randint(2, 4), rnd.randint(2, 8))
                u0, v0 = rnd.randint(0, max(0, gh - bh)), rnd.randint(0, max(0, gw - bw))
                cells |= {u * gw + v for u in range(u0, min(gh, u0 + bh)) for v in range(v0, min(gw, v0 + bw))}
            at = torch.tensor(sorted(cells), device="cuda")
            frame[:, at] = 3.0 * qhat[:, None] + 0.1 * _normal(gen, (L, len(cells), hkv, D))
            if case["exact_dups"] and rnd.random() < 0.4:
                copies = rnd.randint(1, 4)
        k[:, off:off + size] = frame
        end = off + size + case["text"]
        if end > off + size:
            k[:, off + size:end] = _normal(gen, (L, end - off - size, hkv, D), heavy)
        prev = frame
    return k


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _raw(t):
    """The tensor's bit pattern: copied rows are compared as whole values."""
    return t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def _params(case):
    return stlite.make_params(case["beta"], css_size=case["css"], tsg_enable=case["tsg"])


def prepare(case, seed):
    gen, rnd = _gen(seed), random.Random(seed)
    dt, hq, hkv = DTYPES[case["dtype"]], case["hq"], case["hkv"]
    s = dict(case=case)
    if case["kind"] == "decode":
        L, n, w = case["layers"], case["n"], case["w"]
        s["q"] = torch.randn((L, w, hq, D), generator=gen, device="cuda").to(dt)
        s["k"] = torch.randn((L, n, hkv, D), generator=gen, device="cuda").to(dt)
        s["v"] = torch.randn((L, n, hkv, D), generator=gen, device="cuda").to(dt)
        s["out"] = torch.empty((L, w, hq, D), device="cuda")
        sh = stlite.make_shape(s["q"][0], s["k"][0])
        size = stlite.stlite_decode_workspace_size(sh) if L == 1 else stlite.stlite_decode_layers_workspace_size(sh, L)
        s["io"] = [(s["q"][l], s["k"][l], s["v"][l], s["out"][l]) for l in range(L)]
    elif case["kind"] == "prompt":
        s["q"] = torch.randn((case["rows"], hq, D), generator=gen, device="cuda").to(dt)
        s["k"] = torch.randn((case["n"], hkv, D), generator=gen, device="cuda").to(dt)
        s["a"] = torch.empty((hkv, case["n"]), device="cuda")
        size = stlite.stlite_prompt_workspace_size(stlite.prompt_shape(s["q"], s["k"]), case["rows"])
    else:
        L, w, lay = case["layers"], case["w"], _layouts(case)
        S = len(lay)
        q = torch.randn((L, S, w, hq, D), generator=gen, device="cuda").to(dt)
        k = torch.cat([_keys(case, fr, n, q[:, i], gen, rnd) for i, (fr, n) in enumerate(lay)], 1)
        v = torch.randn(k.shape, generator=gen, device="cuda", dtype=dt)
        B = [stlite.stlite_budget(n, case["beta"]) for _, n in lay]
        s["frames"] = [stlite.FrameSpec(*fr) for fr, _ in lay]
        s["params"], s["budget"] = _params(case), B[0]
        s["cu"] = np.concatenate([[0], np.cumsum([n for _, n in lay])]).astype(np.int32)
        s["k_out"] = torch.empty((L, sum(B), hkv, D), dtype=dt, device="cuda")
        s["v_out"] = torch.empty_like(s["k_out"])
        s["idx"] = torch.empty((L, hkv * sum(B)), dtype=torch.int32, device="cuda")
        sh = stlite.make_shape(q[0, 0], k[0])
        if S > 1:
            size = L * stlite.stlite_workspace_size_varlen(sh, s["cu"], s["frames"], s["params"])
        else:
            size = L * stlite.stlite_workspace_size(sh, s["frames"][0], s["params"])
            q = q[:, 0]
        s["q"], s["k"], s["v"] = q, k, v
        s["io"] = [(q[l], k[l], v[l], s["k_out"][l], s["v_out"][l], s["idx"][l]) for l in range(L)]
        n = k.shape[1]
        if case["kind"] == "maps":
            s["a"], s["rho"], s["phi"] = (torch.empty((hkv, n), device="cuda") for _ in range(3))
            s["gate"], s["tau"] = torch.empty((hkv, n), dtype=torch.uint8, device="cuda"), torch.empty(hkv, device="cuda")
        if case["kind"] == "pick":
            # maps as the pass has them: a softmax-mass score, saliencies around 1, text without one,
            # a fifth of the screenshots' tokens behind an open gate
            s["a"] = torch.randn((hkv, n), generator=gen, device="cuda").exp_() * (w / n / 1.6487)
            s["phi"] = (1.0 - 0.09 * torch.randn((hkv, n), generator=gen, device="cuda")).clamp_(0, 2)
            s["gate"] = (torch.rand((hkv, n), generator=gen, device="cuda") < case["beta"]).to(torch.uint8)
            text = torch.ones(n, dtype=torch.bool, device="cuda")
            for off, gh, gw in zip(*lay[0][0]):
                text[off:off + gh * gw] = False
            s["phi"][:, text], s["gate"][:, text] = math.nan, 1
            s["idx"], s["score"] = s["idx"].view(hkv, -1), torch.empty((hkv, n), device="cuda")
    s["ws"] = torch.zeros(size, dtype=torch.uint8, device="cuda")
    return s


# -------------------------------------------------------------------- runs

def run(s):
    case = s["case"]
    if case["kind"] == "decode":
        if case["layers"] == 1:
            stlite.stlite_decode_attention(*s["io"][0], s["ws"])
        else:
            stlite.stlite_decode_attention_layers(s["io"], s["ws"])
        return s["out"]
    if case["kind"] == "prompt":
        base = stlite.STLITE_PROMPT_MEAN if case["mean"] else stlite.STLITE_PROMPT_FULL
        stlite.stlite_prompt_score(s["q"], s["k"], base, s["a"], s["ws"])
        return s["a"]
    q, k, v, fr, ws = s["q"], s["k"], s["v"], s["frames"][0], s["ws"]
    if case["kind"] == "maps":
        stlite.stlite_score(q[0], k[0], s["a"], ws)
        stlite.stlite_gate_frames(q[0], k[0], fr, s["budget"], s["rho"], s["tau"], s["gate"], ws)
        if case["css"] == 3:
            stlite.stlite_spatial_saliency(q[0], k[0], fr, s["phi"], ws)
        else:
            stlite.stlite_spatial_saliency_size(q[0], k[0], fr, case["css"], s["phi"], ws)
        return dict(a=s["a"], rho=s["rho"], tau=s["tau"], gate=s["gate"], phi=s["phi"])
    if case["kind"] == "pick":
        stlite.stlite_select_topk(q[0], k[0], fr, s["params"], s["a"], s["phi"], s["gate"], s["budget"], s["idx"],
                                  s["score"], ws)
        stlite.stlite_compact(q[0], k[0], v[0], s["budget"], s["idx"], s["k_out"][0], s["v_out"][0])
        return dict(idx=s["idx"], k=_raw(s["k_out"]), v=_raw(s["v_out"]), score=s["score"])
    if case["seqs"] > 1:
        stlite.stlite_compress_varlen_layers(s["io"], s["cu"], s["frames"], s["params"], ws)
    elif case["layers"] > 1:
        stlite.stlite_compress_layers(s["io"], fr, s["params"], ws)
    else:  # the convenience call: it makes the outputs
        ko, vo, idx = stlite.compress_layer(q[0], k[0], v[0], fr, beta=case["beta"], css_size=case["css"],
                                            tsg_enable=case["tsg"], ws=ws)
        return dict(idx=idx, k=_raw(ko), v=_raw(vo))
    return dict(idx=s["idx"], k=_raw(s["k_out"]), v=_raw(s["v_out"]))


def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    hq, hkv = case["hq"], case["hkv"]
    if case["kind"] == "decode":
        L, n, w = case["layers"], case["n"], case["w"]
        return dict(bytes=L * (2 * n * hkv * D * e + w * hq * D * (e + 4)), flops=L * 4.0 * w * hq * n * D)
    if case["kind"] == "prompt":
        n, r = case["n"], case["rows"]
        pairs = r * (n - r) + r * (r + 1) / 2
        return dict(bytes=(n * hkv + r * hq) * D * e + 4 * hkv * n, flops=2.0 * pairs * hq * D)
    byts = flops = 0.0
    for (off, gh, gw), n in _layouts(case):
        size = (gh.astype(np.int64) * gw)
        cur, hist = int(size[-1]), int(size[:-1].sum())
        B = stlite.stlite_budget(n, case["beta"])
        row = hkv * D * e
        if case["kind"] == "pick":
            byts += 13 * hkv * n + 4 * row * B + 4 * hkv * B
            flops += 2.0 * hkv * n
            continue
        byts += n * row + case["w"] * hq * D * e
        flops += 2.0 * case["w"] * hq * n * D + 10.0 * (cur + hist) * hkv * D
        if case["tsg"] or case["kind"] == "maps":
            flops += 2.0 * hist * cur * hkv * D
        byts += 13 * hkv * n if case["kind"] == "maps" else 3 * row * B + 4 * hkv * B
    return dict(bytes=byts * case["layers"], flops=flops * case["layers"])


def tolerance(case):
    """About four times the distance from exact() over the ranges of draw()."""
    if case["kind"] == "pick":
        return "exact"
    if case["kind"] == "compress":
        # whole values (indices, copied rows): a token may change places with another whose fp32 score is as
        # close to the threshold as rounding, which moves the rows between the two
        return {"differ": 0.01}
    if case["kind"] == "maps":  # fp32 sums (a: 3e-7 off, largest 2.6e-6; rho 1.6e-7; phi 5e-8); gate: near ties of rho
        return {"rel": 1.2e-6, "max": 1e-5, "differ": 1e-3}
    if case["kind"] == "decode":  # bf16 caches multiply probabilities as two bf16 parts: 2e-6 off, largest 8.5e-6
        return {"rel": 8e-6, "max": 4e-5}
    return {"rel": 1.2e-6, "max": 1e-5}  # prompt, as the score of maps


# ------------------------------------------------------- the same in 64 bits

def _score64(q, k):
    w, hq, _ = q.shape
    n, hkv, _ = k.shape
    q, a = q.double().view(w, hkv, hq // hkv, D), torch.empty((hkv, n), dtype=torch.float64, device="cuda")
    for h in range(hkv):
        x = q[:, h].reshape(-1, D) @ k[:, h].double().T / math.sqrt(D)
        a[h] = torch.softmax(x, 1).sum(0) / (hq // hkv)
    return a


def _gate64(k, frames, budget):
    n, hkv, _ = k.shape
    rho = torch.full((hkv, n), math.nan, dtype=torch.float64, device="cuda")
    tau, gate = torch.full((hkv,), math.nan, dtype=torch.float64, device="cuda"), torch.ones((hkv, n), dtype=torch.uint8, device="cuda")
    spans = [(int(o), int(o + a * b)) for o, a, b in zip(*frames)]
    pool = torch.cat([torch.arange(a, b, device="cuda") for a, b in spans[:-1]] or [torch.arange(0, device="cuda")])
    for h in range(hkv if len(pool) else 0):
        x = k[:, h].double()
        x = x / x.norm(dim=1, keepdim=True).clamp_min(1e-8)
        cur = x[spans[-1][0]:spans[-1][1]].T
        r = torch.cat([(x[p] @ cur).amax(1) for p in pool.split(16384)])
        rho[h, pool] = r
        tau[h] = r.kthvalue(min(budget, len(pool))).values
        gate[h, pool] = (r <= tau[h]).to(torch.uint8)
    return rho, tau, gate


def _phi64(k, frames, size):
    n, hkv, _ = k.shape
    phi = torch.full((hkv, n), math.nan, dtype=torch.float64, device="cuda")
    R = size // 2
    for off, gh, gw in zip(*(x.tolist() for x in frames)):
        x = k[off:off + gh * gw].double()
        x = (x / x.norm(dim=-1, keepdim=True).clamp_min(1e-8)).view(gh, gw, hkv, D)
        pad = torch.zeros((gh + 2 * R, gw + 2 * R, hkv, D), dtype=torch.float64, device="cuda")
        pad[R:R + gh, R:R + gw] = x
        ones = torch.zeros(pad.shape[:2], dtype=torch.float64, device="cuda")
        ones[R:R + gh, R:R + gw] = 1
        tot, cnt = torch.zeros_like(x), torch.zeros((gh, gw), dtype=torch.float64, device="cuda")
        for du in range(size):
            for dv in range(size):
                if (du, dv) != (R, R):
                    tot += pad[du:du + gh, dv:dv + gw]
                    cnt += ones[du:du + gh, dv:dv + gw]
        p = 1 - (x * tot).sum(-1) / cnt.clamp_min(1)[..., None]
        phi[:, off:off + gh * gw] = torch.where(cnt[..., None] > 0, p, 0).view(-1, hkv).T
    return phi


def _visual(frames, n):
    m = torch.zeros(n, dtype=torch.bool, device="cuda")
    for off, gh, gw in zip(*(x.tolist() for x in frames)):
        m[off:off + gh * gw] = True
    return m


def _pick64(a, phi, gate, frames, budget):
    """S of every token and the kept indices in ascending order (equal scores: lower index first)."""
    s = torch.where(_visual(frames, a.shape[1]), torch.where(gate.bool(), a + phi, 0), a)
    keep = torch.sort(s, dim=1, descending=True, stable=True).indices[:, :budget]
    return s, keep.sort(1).values.to(torch.int32)


def _rows(x, idx):
    """x [n][Hkv][d] gathered at idx [Hkv][B] -> [B][Hkv][d]."""
    return x.gather(0, idx.long().T[..., None].expand(-1, -1, D))


def exact(case, seed):
    s = prepare(case, seed)
    q, k = s["q"], s["k"]
    if case["kind"] == "decode":
        L, w, hq, _ = q.shape
        out = torch.empty((L, w, hq, D), dtype=torch.float64, device="cuda")
        G = hq // case["hkv"]
        for l in range(L):
            for g in range(hq):
                p = torch.softmax(q[l, :, g].double() @ k[l, :, g // G].double().T / math.sqrt(D), 1)
                out[l, :, g] = p @ s["v"][l, :, g // G].double()
        return out
    if case["kind"] == "prompt":
        r, n, hkv, G = case["rows"], case["n"], case["hkv"], case["hq"] // case["hkv"]
        a, pos = torch.zeros((hkv, n), dtype=torch.float64, device="cuda"), torch.arange(n, device="cuda")
        for h in range(hkv):
            kh = k[:, h].double().T
            for g in range(h * G, (h + 1) * G):
                for r0 in range(0, r, 2048):
                    x = q[r0:r0 + 2048, g].double() @ kh / math.sqrt(D)
                    p = n - r + r0 + torch.arange(len(x), device="cuda")
                    a[h] += torch.softmax(x.masked_fill_(pos[None] > p[:, None], -math.inf), 1).sum(0)
        a /= G
        return a / torch.clamp(n - pos, max=r) if case["mean"] else a
    lay = _layouts(case)
    fr, n = lay[0]
    if case["kind"] == "maps":
        rho, tau, gate = _gate64(k[0], fr, s["budget"])
        return dict(a=_score64(q[0], k[0]), rho=rho, tau=tau, gate=gate, phi=_phi64(k[0], fr, case["css"]))
    if case["kind"] == "pick":
        score, idx = _pick64(s["a"].double(), s["phi"].double(), s["gate"], fr, s["budget"])
        return dict(idx=None, k=None, v=None, score=score)  # equal fp32 scores may differ in 64 bits
    idx_all, k_all, v_all = [], [], []
    for l in range(case["layers"]):
        for i, (fr, n) in enumerate(lay):
            at = int(s["cu"][i])
            ql = q[l, i] if case["seqs"] > 1 else q[l]
            kl, vl = k[l, at:at + n], s["v"][l, at:at + n]
            b = stlite.stlite_budget(n, case["beta"])
            gate = _gate64(kl, fr, b)[2] if case["tsg"] else torch.ones((case["hkv"], n), device="cuda")
            _, idx = _pick64(_score64(ql, kl), _phi64(kl, fr, case["css"]), gate, fr, b)
            idx_all.append(idx.reshape(-1))
            k_all.append(_rows(kl, idx))
            v_all.append(_rows(vl, idx))
    L = case["layers"]
    idx, ko, vo = torch.cat(idx_all).view(L, -1), torch.cat(k_all), torch.cat(v_all)
    if case["seqs"] == 1 and L == 1:
        return dict(idx=idx.view(case["hkv"], -1), k=_raw(ko), v=_raw(vo))
    return dict(idx=idx, k=_raw(ko.view(L, -1, case["hkv"], D)), v=_raw(vo.view(L, -1, case["hkv"], D)))

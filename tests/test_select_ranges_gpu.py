"""The selection kernel's range passes and its cluster sizes, through
stlite_select_topk against the exact order (no frames, so S = A): score
ranges that put few, many or nearly all keys into the chosen bin (32, 33,
1,024 and 1,025 keys in it are its branches' edges), ranges over the whole
exponent, thresholds at, above and below the zeros that a closed gate
leaves, infinities, and (heads, tokens) that take one CTA, small, odd and
16-CTA clusters, with and without 16-byte rows.  And the fused gate, which
stops at a set instead of a threshold, against the staged maps on keys whose
similarities are units in the last place apart.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import build
    build.build()
    from paper_2603_00188_gb300 import stlite
    return stlite


def _scores(kind, h, n, rng):
    if kind == "exponents":  # every exponent, both signs
        return (rng.choice([-1.0, 1.0], (h, n)) * 2.0 ** rng.uniform(-140, 120, (h, n))).astype(np.float32)
    if kind == "crowd_and_outliers":  # most keys in one bin of the range
        x = (1.0 + 1e-3 * rng.standard_normal((h, n))).astype(np.float32)
        x[:, ::17] = (2.0 ** rng.uniform(-100, 100, x[:, ::17].shape)).astype(np.float32)
        return x
    if kind.startswith("bin_of_"):  # that many keys within a 1,024th of the range, the others spread above and below
        c = min(int(kind[7:]), n // 2)
        x = np.where(rng.random((h, n)) < 0.5, rng.uniform(1.0, 1.4, (h, n)), rng.uniform(1.6, 2.0, (h, n)))
        for i in range(h):
            x[i, rng.permutation(n)[:c]] = 1.5 + 1e-4 * rng.random(c)
        return x.astype(np.float32)
    if kind == "mostly_zero":
        x = rng.standard_normal((h, n)).astype(np.float32)
        x[rng.random((h, n)) < 0.6] = 0.0
        return x
    if kind == "infinities":
        return rng.choice(np.array([np.inf, -np.inf, 0.0, 1.0, 3.4e38], np.float32), (h, n))
    raise ValueError(kind)


KINDS = ["exponents", "crowd_and_outliers", "bin_of_32", "bin_of_33", "bin_of_1024", "bin_of_1025", "mostly_zero",
         "infinities"]
SIZES = [(1, 5), (3, 40), (4, 1152), (112, 2144), (4, 23680), (56, 6001), (4, 132800)]


def _check(st, a, budgets):
    h, n = a.shape
    q = torch.zeros((1, h, 128), dtype=torch.bfloat16, device="cuda")
    k = torch.zeros((n, h, 128), dtype=torch.bfloat16, device="cuda")
    none, a_d, order = ([], [], []), torch.from_numpy(a).cuda(), None
    sh = st.make_shape(q, k)
    for b in budgets:
        prm = st.make_params(1.0, k_override=b, alpha=0.0, tsg_enable=0, css_enable=0)
        ws = st.workspace(sh, none, prm)
        idx = torch.empty((h, b), dtype=torch.int32, device="cuda")
        st.stlite_select_topk(q, k, none, prm, a_d, None, None, b, idx, None, ws)
        if order is None:  # by value, equal ones by index (-0.0 equal to 0.0)
            order = torch.sort(a_d + 0.0, dim=1, descending=True, stable=True).indices
        want = order[:, :b].sort(1).values.to(torch.int32)
        assert torch.equal(idx, want), "budget %d" % b


@pytest.mark.parametrize("h,n", SIZES)
@pytest.mark.parametrize("kind", KINDS)
def test_topk_over_ranges(st, kind, h, n):
    a = _scores(kind, h, n, np.random.default_rng(n + 7 * h + len(kind)))
    _check(st, a, sorted({1, max(1, n // 5), max(1, n // 2), max(1, n - n // 8), n}))


@pytest.mark.parametrize("layers,heads,n", [(1, 4, 2000), (32, 4, 700), (5, 4, 9000), (32, 2, 5000), (11, 1, 3001)])
def test_fused_gate_equals_staged_on_near_duplicates(st, layers, heads, n):
    # frame 1 is frame 0 with noise: the cosines of frame 0 lie within about a thousand ulps
    rng = np.random.default_rng(n)
    gh, gw, w = 16, (n // 2) // 16, 2
    params, ios = st.make_params(0.2), []
    fs = st.FrameSpec([0, gh * gw], [gh, gh], [gw, gw])
    b = st.stlite_budget(n, 0.2)
    for _ in range(layers):
        base = torch.from_numpy(rng.standard_normal((gh * gw, heads, 128), dtype=np.float32)).cuda()
        k = torch.randn((n, heads, 128), device="cuda")
        k[:gh * gw], k[gh * gw:2 * gh * gw] = base, base + 0.01 * torch.randn_like(base)
        k = k.to(torch.bfloat16)
        q = torch.randn((w, heads, 128), device="cuda").to(torch.bfloat16)
        ko = torch.empty((b, heads, 128), dtype=torch.bfloat16, device="cuda")
        ios.append((q, k, k, ko, torch.empty_like(ko), torch.empty((heads, b), dtype=torch.int32, device="cuda")))
    ws = torch.zeros(layers * st.stlite_workspace_size(st.make_shape(q, k), fs, params), dtype=torch.uint8, device="cuda")
    st.stlite_compress_layers(ios, fs, params, ws)
    a, phi, rho = (torch.empty((heads, n), device="cuda") for _ in range(3))
    tau, gate = torch.empty(heads, device="cuda"), torch.empty((heads, n), dtype=torch.uint8, device="cuda")
    for q, k, _, _, _, idx in ios:
        st.stlite_score(q, k, a, ws)
        st.stlite_gate_frames(q, k, fs, b, rho, tau, gate, ws)
        st.stlite_spatial_saliency(q, k, fs, phi, ws)
        want = torch.empty_like(idx)
        st.stlite_select_topk(q, k, fs, params, a, phi, gate, b, want, None, ws)
        assert torch.equal(gate[:, :gh * gw].bool(), rho[:, :gh * gw] <= tau[:, None])
        assert torch.equal(idx, want)

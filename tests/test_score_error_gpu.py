"""How far the base scores are from 64 bits, root mean square.

The other tests allow what a selection can bear, a thousand times the error
that the kernels have.  Here each case states the error measured over its
seeds, and the bound lies between that and what the cheaper forms of the same
sums give, so that going back to one of them shows: the running maximum
itself in the place of a whole number (fp32; 1.3 to 6 times the error, as the
rescaled sums are rounded), plain sums of tiles, groups and CTAs (1.2 to 2.1
times), the rounding errors dropped where sums are merged (1.1 times).  Few
rows, key tiles shared by a cluster, and one CTA per tile are among them.
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

F32, BF16 = torch.float32, torch.bfloat16
SEEDS = 6
# (dtype, keys, window rows, query heads, KV heads), measured, bound
SCORE = [((F32, 300, 32, 28, 4), 4.69e-8, 4.85e-8),
         ((F32, 1152, 1, 28, 4), 2.06e-7, 2.35e-7),
         ((F32, 1152, 64, 28, 4), 3.58e-8, 3.8e-8),
         ((F32, 11840, 32, 28, 4), 7.02e-8, 8.8e-8),
         ((BF16, 300, 32, 28, 4), 6.11e-8, 7.4e-8),
         ((BF16, 1152, 1, 28, 4), 2.35e-7, 2.8e-7),
         ((BF16, 11840, 32, 28, 4), 1.50e-7, 1.9e-7)]
# (dtype, keys, prompt rows, query heads, KV heads)
PROMPT = [((F32, 300, 100, 28, 4), 3.22e-8, 3.45e-8),
          ((F32, 1152, 1, 28, 4), 2.06e-7, 2.35e-7),
          ((F32, 1152, 1152, 28, 4), 2.76e-8, 2.9e-8),
          ((F32, 4000, 1333, 12, 2), 2.28e-8, 2.45e-8),
          ((BF16, 300, 300, 28, 4), 3.61e-8, 4.2e-8),
          ((BF16, 1152, 1, 28, 4), 2.18e-7, 2.7e-7),
          ((BF16, 1152, 1152, 28, 4), 3.78e-8, 3.95e-8),
          ((BF16, 4000, 1333, 12, 2), 4.88e-8, 5.4e-8)]


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import build
    build.build()
    from paper_2603_00188_gb300 import stlite
    return stlite


def inputs(seed, rows, n, hq, hkv, dt):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn((rows, hq, 128), generator=g).to(dt).cuda(),
            torch.randn((n, hkv, 128), generator=g).to(dt).cuda())


def exact(q, k, causal):
    """The attention mass per key, averaged over each KV head's query heads."""
    rows, n, G = q.shape[0], k.shape[0], q.shape[1] // k.shape[1]
    out = torch.zeros((k.shape[1], n), dtype=torch.float64, device="cuda")
    seen = torch.arange(n, device="cuda") <= torch.arange(n - rows, n, device="cuda")[:, None]
    for h in range(q.shape[1]):
        x = q[:, h].double() @ k[:, h // G].double().T / math.sqrt(128)
        if causal:
            x.masked_fill_(~seen, -math.inf)
        out[h // G] += torch.softmax(x, -1).sum(0) / G
    return out


def error(a, ref):
    return float((a.double() - ref).norm() / ref.norm())


@pytest.mark.parametrize("shape,measured,bound", SCORE)
def test_window_score(st, shape, measured, bound):
    dt, n, w, hq, hkv = shape
    err = 0.0
    for seed in range(SEEDS):
        q, k = inputs(seed, w, n, hq, hkv, dt)
        a = torch.empty((hkv, n), device="cuda")
        size = st.stlite_workspace_size(st.make_shape(q, k), st.FrameSpec([], [], []), st.make_params(0.2))
        st.stlite_score(q, k, a, torch.zeros(size, dtype=torch.uint8, device="cuda"))
        err += error(a, exact(q, k, False)) / SEEDS
    assert err <= bound, (err, measured)


@pytest.mark.parametrize("shape,measured,bound", PROMPT)
def test_prompt_base(st, shape, measured, bound):
    dt, n, rows, hq, hkv = shape
    err = 0.0
    for seed in range(SEEDS):
        q, k = inputs(seed, rows, n, hq, hkv, dt)
        a, _ = st.prompt_score(q, k, st.STLITE_PROMPT_FULL)
        err += error(a, exact(q, k, True)) / SEEDS
    assert err <= bound, (err, measured)

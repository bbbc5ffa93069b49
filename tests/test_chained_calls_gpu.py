"""Calls that follow one another on a stream at once, in the same buffers.

Compaction reads the indices that the selection before it is still writing
when compaction's first CTAs arrive, and a decode call may take the previous
call's output as its queries.  Both kernels are launched ahead of their
predecessors, so each must wait for them and read what they wrote, also when
the same memory held other values a moment earlier.  The calls are queued
behind a few milliseconds of other work and run without gaps; the results are
those of the same calls with a synchronisation between them, bit for bit.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

ROUNDS = 24


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import build
    build.build()
    from paper_2603_00188_gb300 import stlite
    return stlite


@pytest.fixture(scope="module")
def filler():
    return torch.zeros(1 << 28, device="cuda")  # 1 GiB


def both_ways(call, rounds, filler):
    """call(i) enqueues round i and returns its outputs' buffers: the copies
    of them with a synchronisation around every round, and without one."""
    out = []
    for sync in (True, False):
        if not sync:
            for _ in range(20):
                filler.add_(1.0)
        got = []
        for i in range(rounds):
            bufs = call(i)
            if sync:
                torch.cuda.synchronize()
            got.append([b.clone() for b in bufs])
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        out.append(got)
    return out


@pytest.mark.parametrize("n,dtype", [(61, torch.float32), (1155, torch.bfloat16), (20000, torch.bfloat16)])
def test_select_then_compact_on_one_index_buffer(st, filler, n, dtype):
    hkv, d, budget = 4, 128, max(1, n // 5)
    g = torch.Generator(device="cuda").manual_seed(n)
    q = torch.randn((8, hkv * 7, d), generator=g, device="cuda").to(dtype)
    k = torch.randn((n, hkv, d), generator=g, device="cuda").to(dtype)
    v = torch.randn((n, hkv, d), generator=g, device="cuda").to(dtype)
    a = (torch.rand((ROUNDS, hkv, n), generator=g, device="cuda").argsort(-1) + 1).float()  # distinct
    frames = ([0], [5], [n // 10])
    prm = st.make_params(0.2, css_enable=0)
    idx = torch.zeros((hkv, budget), dtype=torch.int32, device="cuda")
    base, score = torch.empty((hkv, n), device="cuda"), torch.empty((hkv, n), device="cuda")
    ko = torch.empty((budget, hkv, d), dtype=dtype, device="cuda")
    vo = torch.empty_like(ko)
    ws = torch.zeros(st.stlite_workspace_size(st.make_shape(q, k), frames, prm), dtype=torch.uint8, device="cuda")

    def call(i):
        base.copy_(a[i])
        st.stlite_select_topk(q, k, frames, prm, base, None, None, budget, idx, score, ws)
        st.stlite_compact(q, k, v, budget, idx, ko, vo)
        return idx, ko, vo

    apart, together = both_ways(call, ROUNDS, filler)
    for i, (x, y) in enumerate(zip(apart, together)):
        for p, r in zip(x, y):
            assert torch.equal(p, r), i
        rows = torch.sort(torch.topk(a[i], budget, dim=1).indices, 1).values.to(torch.int32)
        assert torch.equal(y[0], rows), i
        for h in range(hkv):
            assert torch.equal(y[1][:, h], k[rows[h].long(), h]) and torch.equal(y[2][:, h], v[rows[h].long(), h])


@pytest.mark.parametrize("n", [33, 4097])
def test_fp32_decode_on_the_previous_output(st, filler, n):
    hq, hkv, d = 28, 4, 128
    g = torch.Generator(device="cuda").manual_seed(n)
    k = torch.randn((n, hkv, d), generator=g, device="cuda")
    v = 6.0 * torch.randn((n, hkv, d), generator=g, device="cuda")
    start = torch.randn((1, hq, d), generator=g, device="cuda")
    q = [start.clone(), torch.zeros_like(start)]  # each call reads one and writes the other
    ws = torch.zeros(st.stlite_decode_workspace_size(st.make_shape(start, k)), dtype=torch.uint8, device="cuda")

    def call(i):
        if i == 0:
            q[0].copy_(start)
        for _ in range(4):
            st.stlite_decode_attention(q[0], k, v, q[1], ws)
            st.stlite_decode_attention(q[1], k, v, q[0], ws)
        return q

    apart, together = both_ways(call, ROUNDS, filler)
    for i, (x, y) in enumerate(zip(apart, together)):
        assert torch.equal(x[0], y[0]) and torch.equal(x[1], y[1]), i
    kk, vv = k.double().repeat_interleave(hq // hkv, 1), v.double().repeat_interleave(hq // hkv, 1)
    x = together[0][0].double()
    p = torch.softmax(torch.einsum("whd,nhd->whn", x, kk) / d ** 0.5, -1)
    out = torch.empty_like(start)
    st.stlite_decode_attention(together[0][0], k, v, out, ws)
    # a score's rounding error (128 fp32 products of values up to ~100, over
    # sqrt(128)) is below 5e-5, and moves the weights by as much, relatively
    assert torch.allclose(out.double(), torch.einsum("whn,nhd->whd", p, vv), rtol=0, atol=1e-4 * float(v.abs().max()))

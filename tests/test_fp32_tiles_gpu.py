"""The fp32 passes (64 x 64 tiles of dot products) at the edges of their
tiles: query rows, keys, historical tokens and current-frame columns one
below, at and one above a tile, empty key splits, one-token frames and
several column slices, against the fp64 oracle under the parity rules."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_00188_gb300 import synth
from parity import a_bound, assert_within, cos_bound, exact64, pool_mask, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import build
    build.build()
    from paper_2603_00188_gb300 import stlite
    return stlite


# (w, hq, hkv, text, grids): R = w hq / hkv query rows; the last grid is the
# current frame, the others the TSG pool
CASES = {
    "one_tile": (32, 4, 2, 1, [(8, 8), (8, 8)]),                     # R = 64, 64 x 64 tokens
    "one_below": (9, 14, 2, 3, [(7, 9), (9, 7)]),                    # R = 63, 63-token frames
    "one_above": (13, 5, 1, 0, [(5, 13), (13, 5), (5, 13)]),         # R = 65, 65-token frames
    "one_token_frames": (1, 2, 2, 2, [(1, 1), (1, 1)]),              # R = 1, N = 6
    "half_row_tiles": (3, 4, 2, 5, [(3, 43), (12, 16), (1, 64), (1, 129)]),  # 129, 192, 64 | 129
    "two_slices_full": (4, 4, 1, 7, [(8, 8), (16, 16)]),             # four column tiles, one CTA row
    "ragged_slices": (64, 8, 1, 11, [(10, 13), (17, 19)]),           # R = 512, 323 columns
    "wide_current": (2, 2, 1, 0, [(2, 3), (30, 41)]),                # 6 rows against 1,230 columns
}


@pytest.mark.parametrize("name", list(CASES))
def test_fp32_tiles(st, name):
    w, hq, hkv, text, grids = CASES[name]
    rng = np.random.default_rng(len(name))
    offs, at = [], 0
    for gh, gw in grids:
        offs.append(at)
        at += gh * gw + text
    n = at
    k = rng.standard_normal((n, hkv, 128), dtype=np.float32)
    wl = synth.Workload(name, rng.standard_normal((w, hq, 128), dtype=np.float32), k, k.copy(),
                        np.array(offs, np.int32), np.array([g[0] for g in grids], np.int32),
                        np.array([g[1] for g in grids], np.int32), beta=0.3, dtype="f32")
    q, kd, _ = to_device(wl)
    sh = st.make_shape(q, kd)
    ws = st.workspace(sh, wl.frames)
    a = torch.empty((hkv, n), device="cuda")
    rho, tau = torch.empty_like(a), torch.empty(hkv, device="cuda")
    gate = torch.empty((hkv, n), dtype=torch.uint8, device="cuda")
    b = oracle.budget(n, 0.3)
    st.stlite_score(q, kd, a, ws)
    st.stlite_gate_frames(q, kd, wl.frames, b, rho, tau, gate, ws)
    torch.cuda.synchronize()
    ora = oracle.abase(exact64(q), exact64(kd), threads=4)
    for h in range(hkv):
        assert_within(a[h].cpu().numpy(), ora[h], a_bound(ora[h]), "A_base head %d" % h)
    pool = pool_mask(n, wl.frames)
    rg, ro = rho.cpu().numpy(), oracle.tsg_rho(exact64(kd), wl.frames, threads=4)
    assert np.isnan(rg[:, ~pool]).all()
    assert_within(rg[:, pool], ro[:, pool], cos_bound(ro[:, pool]), "rho")
    assert st.stlite_device_status(ws) == st.STLITE_OK

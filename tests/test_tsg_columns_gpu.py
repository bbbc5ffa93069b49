"""TSG's column halves (bf16): current frames whose columns end one below, at
and one above each 64, 128, 256 and 512, so that a chunk's second stage and a
stage's second half are absent, nearly empty, ragged or full; and pools of
many row tiles, where a last chunk of few columns gets fewer CTAs than the
others; against the fp64 oracle under the parity rules."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_00188_gb300 import synth
from parity import assert_within, cos_bound, exact64, pool_mask, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import build
    build.build()
    from paper_2603_00188_gb300 import stlite
    return stlite


@pytest.mark.parametrize("cols, hist", [(c, (11, 13)) for c in (
    1, 63, 64, 65, 127, 128, 129, 191, 193, 255, 256, 257, 320, 321, 384, 385, 511, 512, 513, 641, 769, 1025)] +
    [(600, (63, 67)), (800, (77, 81)), (1100, (90, 101))])
def test_tsg_columns(st, cols, hist):
    w, hq, hkv, text = 1, 2, 2, 3
    grids = [hist, (1, 129), (1, cols) if cols <= 256 else (cols, 1)]
    offs, at = [], 0
    for gh, gw in grids:
        offs.append(at)
        at += gh * gw + text
    rng = np.random.default_rng(cols)
    k = rng.standard_normal((at, hkv, 128), dtype=np.float32)
    wl = synth.Workload("cols", rng.standard_normal((w, hq, 128), dtype=np.float32), k, k.copy(),
                        np.array(offs, np.int32), np.array([g[0] for g in grids], np.int32),
                        np.array([g[1] for g in grids], np.int32), beta=0.3, dtype="bf16")
    q, kd, _ = to_device(wl)
    ws = st.workspace(st.make_shape(q, kd), wl.frames)
    rho, tau = torch.empty((hkv, at), device="cuda"), torch.empty(hkv, device="cuda")
    gate = torch.empty((hkv, at), dtype=torch.uint8, device="cuda")
    st.stlite_gate_frames(q, kd, wl.frames, oracle.budget(at, 0.3), rho, tau, gate, ws)
    torch.cuda.synchronize()
    pool = pool_mask(at, wl.frames)
    rg, ro = rho.cpu().numpy(), oracle.tsg_rho(exact64(kd), wl.frames, threads=4)
    assert np.isnan(rg[:, ~pool]).all()
    assert_within(rg[:, pool], ro[:, pool], cos_bound(ro[:, pool]), "rho")
    assert st.stlite_device_status(ws) == st.STLITE_OK

"""Phi of text tokens is NaN wherever the text lies: before the first frame,
between frames, after the last one, with gaps longer than a launch's threads,
none at all, and single-cell frames; and Phi of the frames is untouched by it."""
import numpy as np
import pytest
import torch

import oracle
from parity import assert_within, cos_bound, exact64, visual_mask

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,frames", [
    (50, ([0], [5], [10])),                         # no text
    (5000, ([4200], [3], [4])),                     # text before and after one small frame
    (9000, ([1, 20, 8000], [2, 3, 1], [3, 4, 1])),  # gaps of 13 and 7,968 tokens
    (64, ([63], [1], [1])),
])
def test_text_phi_is_nan(n, frames):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_00188_gb300 import stlite as st
    frames = tuple(np.array(x, np.int32) for x in frames)
    gen = torch.Generator().manual_seed(n)
    q = torch.randn((1, 2, 128), generator=gen).to(torch.bfloat16).cuda()
    k = torch.randn((n, 2, 128), generator=gen).to(torch.bfloat16).cuda()
    phi = torch.zeros((2, n), device="cuda")
    st.stlite_spatial_saliency(q, k, frames, phi, st.workspace(st.make_shape(q, k), frames))
    pg, vis = phi.cpu().numpy(), visual_mask(n, frames)
    assert np.isnan(pg[:, ~vis]).all()
    ora = oracle.css_phi(exact64(k), frames, threads=4)
    assert_within(pg[:, vis], ora[:, vis], cos_bound(ora[:, vis]), "Phi")

"""Tensors written between iterations of the quantised method, whose p exists as codes alone."""

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth

pytestmark = pytest.mark.gpu


# levels beyond the largest fp16 value, and levels below the smallest normal one
@pytest.mark.parametrize("scale", [1e5, 1.0, 1e-6])
@pytest.mark.parametrize("kind", [B.T_W, B.T_Z])
@pytest.mark.parametrize("look_at_p", [False, True])
def test_residual_from_scratch_after_quantised_iterations(scale, kind, look_at_p):
    """Writing a tensor back as it is makes the next iteration form r = W p + b - z from the stored tensors.  A twin carries r on:
    both are single-precision values of the same r, so theta_l and W_l of the iteration agree to the rounding of r, at most
    1e-6 of W p, over r itself, not below 1/2 of 1/255 of W p here (the start's projection): 1e-3."""
    inp = synth.make_inputs(synth.small("c2", 700, feat_dim=30, hidden=50, n_layers=4, quant_levels=256))
    inp.features = (inp.features * np.float32(scale)).astype(np.float32)
    got = []
    for rebuild in (False, True):
        ctx = B.from_inputs(inp)
        ctx.step(3)
        if rebuild:
            if look_at_p:
                ctx.get_tensor(B.T_P, 3)
            ctx.set_tensor(kind, 3, ctx.get_tensor(kind, 3))
        ctx.step(1)
        got.append([(ctx.get_tensor(B.T_THETA, l).item(), ctx.get_tensor(B.T_W, l).astype(np.float64)) for l in range(1, 5)])
        ctx.destroy()
    for (t0, w0), (t1, w1) in zip(*got):
        assert abs(t1 - t0) <= 1e-3 * abs(t0)
        assert np.linalg.norm(w1 - w0) <= 1e-3 * np.linalg.norm(w0)

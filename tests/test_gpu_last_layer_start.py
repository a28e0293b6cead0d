"""The last layer's Newton steps start from the stored z; where that does not converge they start again from a."""

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,seed", [(64, 8), (64, 0), (40, 6)])
def test_a_start_far_from_the_root_does_not_cost_the_answer(C, seed):
    """One layer with X = 0: b = 0 at the start, so r = -z, the column mean of z goes to b and a = mean_j z for every node.  The z
    of the labelled nodes are far from it (one unlabelled node carries the mean); of 1199 Newton searches from these z about
    50 do not converge in 100 steps, from a all do.  z is the root of softmax(z) - e_y + nu (z - a) = 0 for the single-precision
    a: |gradient| <= 1e-10, plus what the rounding of z to single precision (d = half a unit in the last place of the node's
    largest |z|) makes of it: nu d, the same again for a, and in the softmax at most a factor e^(2 d) of s_c or of 1 - s_c."""
    n, nu = 1200, np.float32(1e-6)
    inp = synth.make_inputs(synth.small("c2", n, feat_dim=3, n_hops=0, n_layers=1, n_classes=C, quant_levels=0))
    inp.features = np.zeros_like(inp.features)
    rng = np.random.default_rng(seed)
    a = (rng.standard_normal(C) * 1e4).astype(np.float32)
    inp.labels = rng.integers(0, C, n).astype(inp.labels.dtype)
    inp.train_mask = np.ones_like(inp.train_mask)
    inp.train_mask[n - 1] = 0
    z0 = (rng.standard_normal((n, C)) * 30).astype(np.float32)
    z0[n - 1] = n * a.astype(np.float64) - z0[:n - 1].astype(np.float64).sum(0)
    ctx = B.from_inputs(inp, nu=float(nu))
    ctx.set_tensor(B.T_Z, 1, z0)
    ctx.step(1)
    z = ctx.get_tensor(B.T_Z, 1).astype(np.float64)[:n - 1]
    ctx.destroy()
    mean = (z0.astype(np.float64).sum(0) / n).astype(np.float32)
    a = ((-z0 + mean) + z0).astype(np.float64)[:n - 1]
    grad = np.exp(z - z.max(1, keepdims=True))
    grad /= grad.sum(1, keepdims=True)
    d = 0.5 * np.spacing(np.abs(np.concatenate([z, a], 1)).max(1, keepdims=True).astype(np.float32)).astype(np.float64)
    bound = 1e-10 + 2 * float(nu) * d + np.minimum(grad, 1 - grad) * np.expm1(2 * d)
    grad[np.arange(n - 1), inp.labels[:n - 1]] -= 1.0
    grad += float(nu) * (z - a)
    assert np.all(np.abs(grad) <= bound)

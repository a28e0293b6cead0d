"""What an expired wait inside a product leaves behind does not reach the next iteration."""

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth
import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [0, 16, 4096])
@pytest.mark.parametrize("flags", [0, B.FLAG_ONE_LANE | B.FLAG_NO_GRAPH])
def test_leftover_counters_do_not_reach_the_next_iteration(levels, flags):
    inp = synth.make_inputs(synth.small("c2", 600, feat_dim=20, hidden=40, n_layers=4, quant_levels=levels))
    kinds = [(B.T_W, 1, 4), (B.T_B, 1, 4), (B.T_Z, 1, 4), (B.T_Q, 1, 3), (B.T_U, 1, 3), (B.T_P, 2, 4)]
    got = []
    for expired in (False, True):
        ctx = B.from_inputs(inp, flags=flags)
        ctx.step(3)
        if expired:
            assert B.lib().pdadmm_selftest_expired_wait(ctx._h) == B.ETIMEOUT
        for kind, lo, hi in kinds:                 # both form everything derived from the tensors again
            for l in range(lo, hi + 1):
                ctx.set_tensor(kind, l, ctx.get_tensor(kind, l))
        ctx.step(2)
        got.append((U.read_state(ctx), [ctx.get_tensor(B.T_TAU, l).item() for l in (2, 3, 4)]))
        ctx.destroy()
    for k in got[0][0]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0][0][k], got[1][0][k])), k
    assert got[0][1] == got[1][1]

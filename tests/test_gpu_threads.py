"""Contexts in several host threads at once: one captures its iteration into a graph while others come and go."""

import threading

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth

pytestmark = pytest.mark.gpu


def test_contexts_come_and_go_while_another_captures_its_graph():
    inp = synth.make_inputs(synth.small("c2", 300, feat_dim=10, hidden=24, n_layers=8, quant_levels=0))
    want = B.from_inputs(inp)
    want.step(4)
    want_W = want.get_tensor(B.T_W, 3)
    want.destroy()
    errors, ends = [], threading.Event()

    def train():
        try:
            for _ in range(150):
                ctx = B.from_inputs(inp)
                ctx.step(4)
                assert np.array_equal(ctx.get_tensor(B.T_W, 3), want_W)
                ctx.destroy()
        except Exception as e:
            errors.append(e)
        finally:
            ends.set()

    def come_and_go():
        try:
            while not ends.is_set():
                ctx = B.from_inputs(inp)
                ctx.objective()
                ctx.destroy()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=train)] + [threading.Thread(target=come_and_go) for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]

"""The z-update from a lookup table: the chosen candidate against a search over all of them, where the descent can go wrong
(tables of 2 and 3 candidates and of the largest size, minimisers at and beyond the ends of the table, values of q for
which the objective is not convex and all candidates have to be tried)."""

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth
import oracle.pdadmm_oracle as o
import parity_util as U
from test_gpu_parity import _compare_iteration

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act,T,lo,hi,q_scale", [(1, 2, -1.0, 1.0, 0.5), (1, 3, -6.0, 6.0, 1.0), (1, 513, -0.25, 0.25, 1.0),
                                                 (1, 513, -6.0, 6.0, 4.0), (1, 4096, -6.0, 6.0, 1.2), (2, 513, -6.0, 6.0, 1.0),
                                                 (2, 257, -4.0, 4.0, 60.0), (1, 129, -300.0, 300.0, 1.0)])
def test_the_table_candidate_is_the_best_of_all(act, T, lo, hi, q_scale):
    inp = synth.make_inputs(synth.small("c2", 777, feat_dim=9, hidden=37, n_layers=3, quant_levels=0))
    ctx = B.from_inputs(inp, activation=act, table=(T, lo, hi))
    rng = np.random.default_rng(T)
    z0, q0 = {}, {}
    for l in (1, 2):
        z0[l] = rng.standard_normal((777, 37)).astype(np.float32) * np.float32(0.4 * (hi - lo))
        q0[l] = rng.standard_normal((777, 37)).astype(np.float32) * np.float32(q_scale)
        ctx.set_tensor(B.T_Z, l, z0[l])
        ctx.set_tensor(B.T_Q, l, q0[l])
    ctx.step(1)
    step = np.float32(np.float32(hi) - np.float32(lo)) / np.float32(T - 1)
    pts = np.float32(lo) + np.arange(T, dtype=np.float32) * step          # one rounded multiply, one rounded add
    f = np.tanh(pts.astype(np.float64)) if act == 1 else 1.0 / (1.0 + np.exp(-pts.astype(np.float64)))
    for l in (1, 2):
        W, b, p = (ctx.get_tensor(k, l).astype(np.float64) for k in (B.T_W, B.T_B, B.T_P))
        z = ctx.get_tensor(B.T_Z, l)
        a = p @ W.T + b
        at = np.searchsorted(pts, z.ravel()).reshape(z.shape)
        assert np.array_equal(pts[np.minimum(at, T - 1)], z), "z left the table"

        def value(zc, fc):
            return (zc - a) ** 2 + (q0[l] - fc) ** 2 + (zc - z0[l]) ** 2
        got = value(z.astype(np.float64), f[at])
        best = np.full(z.shape, np.inf)
        for i in range(T):
            best = np.minimum(best, value(np.float64(pts[i]), f[i]))
        # a (a product of 27 or 37 terms, kept as r + z in single precision) and the values themselves carry at most
        # 1e-6 of |a| + |z| + |q|: the difference of two values within 2 |d| times that, d the distances that enter them
        size = np.abs(a) + np.abs(z0[l]) + np.abs(q0[l]) + abs(lo) + abs(hi)
        assert np.all(got - best <= 1e-5 * best + 4e-6 * size * (np.sqrt(best) + step))
    ctx.destroy()


@pytest.mark.parametrize("act", [1, 2])
@pytest.mark.parametrize("lo,r,T", [(1e6, 0.3, 78), (7.3e6, 0.1, 66), (3e6, 0.7, 58), (1e6, 4.0, 50), (600.0, 1000.0, 50)])
def test_a_table_finer_than_the_numbers_it_holds(act, lo, r, T):
    """Spacings of r units in the last place of the candidates: neighbouring candidates coincide or lie unevenly, and only a search
    over all of them finds the first smallest one.  With p = 0 every operand is known bit for bit: b = 0 at the start, so
    r = -z, its column mean (a sum that double precision holds exactly) goes to b, a = (r - mean) + z, and f is 1 at such z.
    (The spacing of the last table is resolved: it takes the short search.)"""
    f = np.float32
    n, width = 777, 64
    lo = f(lo)
    hi = f(lo + r * np.spacing(lo) * (T - 1))
    inp = synth.make_inputs(synth.small("c2", n, feat_dim=9, hidden=width, n_layers=2, quant_levels=0))
    inp.features = np.zeros_like(inp.features)
    rng = np.random.default_rng(T)
    col = rng.uniform(lo - 0.3 * (hi - lo), hi + 0.3 * (hi - lo), width).astype(f)
    z0 = (col + np.spacing(lo) * rng.integers(-5, 6, (n, width))).astype(f)
    q0 = (1 + rng.standard_normal((n, width)) * rng.choice([0, 1e-2, 0.3], (n, width))).astype(f)
    ctx = B.from_inputs(inp, activation=act, table=(T, float(lo), float(hi)))
    ctx.set_tensor(B.T_Z, 1, z0)
    ctx.set_tensor(B.T_Q, 1, q0)
    ctx.step(1)
    z = ctx.get_tensor(B.T_Z, 1)
    ctx.destroy()
    step = f(hi - lo) / f(T - 1)
    pts = lo + np.arange(T, dtype=f) * step
    fv = (np.tanh(pts.astype(np.float64)) if act == 1 else 1 / (1 + np.exp(-pts.astype(np.float64)))).astype(f)
    mean = (-z0).astype(np.float64).sum(0) * (1.0 / n)
    a = ((-z0) - mean.astype(f)) + z0

    def fma(x, y, c):
        return (x.astype(np.float64) * y + c).astype(f)      # the product is exact in double precision
    best, want = np.full(z.shape, np.inf, f), np.zeros(z.shape, f)
    for i in range(T):
        d0, d1, d2 = pts[i] - a, q0 - fv[i], pts[i] - z0
        h = fma(d0, d0, fma(d1, d1, d2 * d2))
        want, best = np.where(h < best, pts[i], want), np.minimum(h, best)
    assert np.array_equal(z, want)


# a table without a candidate at zero, and f with f(0) = 1/2; rows of 37 columns lie in rows of 48, of 250 in rows of 256
@pytest.mark.parametrize("name,code,T,hidden,levels,neg,step", [("tanh", 1, 300, 37, 0, 0, 0.0), ("sigmoid", 2, 300, 250, 0, 0, 0.0),
                                                                ("sigmoid", 2, 301, 37, 64, 0, 0.0), ("tanh", 1, 300, 37, 33, 16, 0.0625)])
def test_padding_adds_nothing_to_tau_objective_and_residuals(name, code, T, hidden, levels, neg, step):
    """After three iterations the device's own state goes through one more on both sides: p, tau and the rest as in every parity test;
    then objective and residuals of the state that the device holds.  A squared difference p - q carries 2^-23 |q| / |p - q| of itself: 1e-4
    where p and q agree to three digits."""
    inp = synth.make_inputs(synth.small("c2", 700, feat_dim=9, hidden=hidden, n_layers=4, quant_levels=levels))
    table = (T, -6.0, 6.0)
    prm, prev, _ = U.oracle_problem(inp, neg_levels=neg, step=step, activation=name, table=table)
    ctx = B.from_inputs(inp, quant_neg_levels=neg, quant_step=step, activation=code, table=table)

    def held():
        s = prev.copy()
        for k, v in U.read_state(ctx).items():
            setattr(s, k, v)
        if levels:
            s.scale = [prev.scale[0]] + [float(ctx.get_tensor(B.T_QSCALE, l)[0]) for l in range(2, 5)]
        return s
    ctx.step(3)
    _compare_iteration(ctx, held(), prm, f"{name}/{T}/m={levels}")
    s = held()
    want = o.objective(s, prm)
    assert np.allclose(ctx.objective(), want, rtol=1e-4, atol=1e-6 * abs(want[5]))
    assert np.allclose(ctx.residuals(), o.residuals_sq(s), rtol=1e-4)
    ctx.destroy()

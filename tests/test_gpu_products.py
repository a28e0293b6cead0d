"""The product kernel inside whole iterations where its variants meet their edges: single blocks and pairs of SMs, ragged
tiles, operands whose planes were refused (made again inside the product, or by a kernel beforehand), more layers than one
launch takes; and the last layer's update at the edges of its lanes-per-node rule, host copies at the edges of their pieces."""

import dataclasses

import numpy as np
import pytest

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import synth
import oracle.pdadmm_oracle as o
import error_bounds as E
import parity_util as U
from test_gpu_parity import _compare_iteration

pytestmark = pytest.mark.gpu


# nodes x width: single blocks below three quarters of the pairs (56 tiles of 256 x 128 over the layers of a launch), pairs from
# there on; refused planes are made again beforehand from 2^20 elements on, by the product's own warps below.
@pytest.mark.parametrize("n_nodes,hidden,n_layers", [(131, 68, 4),          # single blocks, split in the product
                                                     (14336 + 3, 64, 6),    # pairs, split in the product
                                                     (4200, 260, 2),        # single blocks, planes made again beforehand
                                                     (8200, 132, 6)])       # pairs, planes made again beforehand
def test_refused_planes_in_every_form_of_the_product(n_nodes, hidden, n_layers):
    """The exponents predicted for the planes of g do not fit where max|g| moves by more than 2^4 up or 2^4 down between
    teacher-forced iterations (predicted is 2^10 .. 2^11, usable are [2^6, 2^15)).  The last layer's does in the second one, from
    rounding noise to its first gradient, and the next layer's in the fourth; u is scaled by 100 and back, which moves the
    others' by 13.  The oracle's gradients say that it is so.  (At 300 the scaled state has 1.2 % of its z at an exact tie of the
    two ReLU candidates, and the comparison allows 1 %.)  Every variable is held to the rounding bounds of its own computation."""
    inp = synth.make_inputs(synth.small("c2", n_nodes, feat_dim=20, hidden=hidden, n_layers=n_layers, quant_levels=0))
    prm, s, _ = U.oracle_problem(inp)
    ctx = B.from_inputs(inp)
    before = None
    for k, factor in enumerate([1.0, 1.0, 100.0, 1 / 100.0]):
        prev = U.round_state(dataclasses.replace(s, u=[x * factor for x in s.u]))
        top = [np.frexp(np.abs(o.grad_p_phi(prev.p[l], prev.W[l], prev.b[l], prev.z[l], prm.nu, prev.q[l - 1], prev.u[l - 1], prm.rho)).max())[1]
               for l in range(1, prev.L)]
        refused = [not 6 <= 10 + now - then <= 14 for now, then in zip(top, before)] if k else []
        if k == 1:
            assert refused[-1]
        if k == 3 and n_layers > 2:
            assert refused[-2]
        before = top
        U.load_state(ctx, prev, False)
        s = _compare_iteration(ctx, prev, prm, f"N={n_nodes}/h={hidden}/k={k}", single_bounds=True)
    ctx.destroy()


@pytest.mark.parametrize("n_layers", [17, 18, 19])                          # 15, 16 and 17 hidden layers: one launch or two
@pytest.mark.parametrize("levels", [0, 16])
def test_grouped_launches_do_not_change_a_bit(n_layers, levels):
    inp = synth.make_inputs(synth.small("c2", 700, feat_dim=30, hidden=72, n_layers=n_layers, quant_levels=levels))
    ref = None
    for flags in (B.FLAG_ONE_LANE | B.FLAG_NO_GRAPH, 0):
        ctx = B.from_inputs(inp, flags=flags)
        ctx.step(2)
        st = U.read_state(ctx)
        ctx.destroy()
        if ref is None:
            ref = st
        else:
            for k in st:
                assert all(np.array_equal(a, b) for a, b in zip(st[k], ref[k])), k


@pytest.mark.parametrize("n_classes", [2, 4, 5, 8, 9, 16, 17, 32, 33, 64])
def test_last_layer_update_at_the_edges_of_its_lanes_per_node(n_classes):
    inp = synth.make_inputs(synth.small("c2", 517, feat_dim=11, hidden=24, n_layers=3, n_classes=n_classes, quant_levels=0))
    prm, s, _ = U.oracle_problem(inp)
    ctx = B.from_inputs(inp)
    for k in range(2):
        prev = U.round_state(s)
        U.load_state(ctx, prev, False)
        s = _compare_iteration(ctx, prev, prm, f"C={n_classes}/k={k}")
    ctx.destroy()


# rows of 1 to 333 values, matrices of a piece (512 KB) and a little less and more
@pytest.mark.parametrize("n_nodes,hidden", [(1, 1), (2047, 64), (2048, 64), (2049, 64), (4000, 333), (131073, 1)])
def test_host_copies_at_the_edges_of_a_piece(n_nodes, hidden):
    inp = synth.make_inputs(synth.small("c2", n_nodes, feat_dim=3, hidden=hidden, n_layers=3, n_hops=1, quant_levels=0))
    ctx = B.from_inputs(inp)
    x = np.random.default_rng(0).standard_normal((n_nodes, hidden)).astype(np.float32)
    ctx.set_tensor(B.T_Z, 1, x)
    assert np.array_equal(ctx.get_tensor(B.T_Z, 1), x)
    ctx.destroy()


# columns at the edges of a wide tile (256) and of its halves, rows at those of a pair's 256 and a block's 128, contractions at those of
# a K block.  Three of the shapes run on wide tiles (the next test has the others of those).
@pytest.mark.parametrize("mode,M,N,K", [(0, 18944, 256, 640), (0, 18945, 255, 641), (1, 19000, 257, 1000), (1, 9600, 500, 703),
                                        (0, 4800, 1025, 1600), (2, 500, 700, 30000), (2, 257, 2049, 16001), (2, 512, 512, 40000)])
def test_wide_tiles_at_their_edges(mode, M, N, K):
    """Every element within LAMBDA standard deviations of KAPPA times the root-sum-square of its terms, the product's bound in the
    iteration tests."""
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((K, M) if mode == 2 else (M, K), dtype=np.float32)
    b = rng.standard_normal((N, K) if mode == 0 else (K, N), dtype=np.float32)
    c, ss = B.matmul(mode, a, b)
    at, bt = (a.T if mode == 2 else a).astype(np.float64), (b.T if mode == 0 else b).astype(np.float64)
    bound = E.LAMBDA * E.kappa(True) * np.sqrt((at ** 2) @ (bt ** 2))
    assert (np.abs(c - at @ bt) <= bound).all()
    assert abs(ss - (c.astype(np.float64) ** 2).sum()) <= 1e-6 * ss


# One round of wide tiles, several, and a last one of a few tiles cut along the contraction (2, 12 or 5 of them, in 2 to 5 slices); over node
# slices; shapes beside them that keep narrow tiles, with the last round cut.
@pytest.mark.parametrize("mode,M,N,K,wide,cut", [
    (0, 18944, 256, 640, True, False), (0, 18690, 255, 641, True, False), (1, 18690, 255, 641, True, False), (0, 9400, 500, 703, True, False),
    (1, 9400, 509, 703, True, False), (0, 9600, 500, 3001, True, True), (1, 4900, 2047, 2049, True, True), (0, 18945, 1025, 2049, True, True),
    (1, 18945, 1025, 1025, True, True), (2, 500, 700, 30000, True, False), (2, 511, 769, 30000, True, False),
    (1, 19000, 257, 1000, False, True), (0, 4800, 1025, 1600, False, True)])
def test_tiles_of_the_form_that_the_shape_is_for(mode, M, N, K, wide, cut):
    before = B.product_forms()
    test_wide_tiles_at_their_edges(mode, M, N, K)
    assert tuple(x - y for x, y in zip(B.product_forms(), before)) == (1, int(wide), int(cut))


def test_refused_planes_on_wide_tiles():
    """The same as above where the product W g runs on wide tiles and splits its refused operands itself (2000 x 500: below 2^20
    elements)."""
    test_refused_planes_in_every_form_of_the_product(2000, 500, 10)


# rows of one group of four columns, of groups that leave lanes of a block idle, of more groups than a block has threads; 8-bit codes
# (integer operands) and 16-bit codes of more levels than those take
@pytest.mark.parametrize("hidden,levels", [(4, 0), (33, 0), (349, 0), (1030, 16), (2050, 0), (100, 4096)])
def test_column_sums_and_unstored_q_at_the_edges_of_a_row(hidden, levels):
    """q is not stored between iterations (q = f(z) + u/nu): what is read back follows from z and u, and setting it to what was read
    -- the next iteration then reads the stored q and applies G p+ in a pass of its own -- changes no bit of the iterates.  The
    iteration in between is the oracle's, with b from the column sums."""
    inp = synth.make_inputs(synth.small("c2", 261, feat_dim=9, hidden=hidden, n_layers=3, quant_levels=levels))
    nu = inp.workload.nu
    got = []
    for set_again in (False, True):
        ctx = B.from_inputs(inp)
        ctx.step(3)
        for l in (1, 2):
            z, u, q = (ctx.get_tensor(k, l) for k in (B.T_Z, B.T_U, B.T_Q))
            f = np.maximum(z, 0)
            assert (np.abs(q - (f + u / np.float32(nu))) <= 4 * 2.0 ** -23 * (np.abs(f) + np.abs(u / nu))).all()
            if set_again:
                ctx.set_tensor(B.T_Q, l, q)
                ctx.set_tensor(B.T_U, l, u)
        ctx.step(2)
        got.append(U.read_state(ctx))
        ctx.destroy()
    for k in got[0]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0][k], got[1][k])), k
    prm, s, _ = U.oracle_problem(inp)
    ctx = B.from_inputs(inp)
    prev = U.round_state(s)
    U.load_state(ctx, prev, levels > 0)
    _compare_iteration(ctx, prev, prm, f"h={hidden}/m={levels}")
    ctx.destroy()


def test_norms_of_many_wide_layers_of_one_tile_each():
    """Thirteen layers of 2000 x 512 in one launch: a pair of SMs has one wide tile of each of up to three layers, and a tile of the norm-only product
    is a single read-out of its accumulator, so warps run ahead of one another by whole layers.  ||W g||^2 of every layer has all of its
    512 parts: a missing one, or one of an earlier product, moves tau by 2e-3 of itself (g from the oracle's formula in 64 bits on the
    device's own state: 1e-5 with one fp16 plane, averaged over 10^6 squares).  Every run gives the same bits."""
    inp = synth.make_inputs(synth.small("c2", 2000, feat_dim=20, hidden=512, n_layers=14, quant_levels=16))
    prm, s, _ = U.oracle_problem(inp)
    bits = []
    for run in range(3):
        ctx = B.from_inputs(inp)
        taus = []
        for it in range(4):
            if run == 0 and it == 3:
                for k, v in U.read_state(ctx).items():
                    setattr(s, k, v)
            before = B.product_forms()
            ctx.step(1)
            # ||W g||^2; the W-gradient and G p+, which take X and integers in launches of their own
            assert B.product_forms()[1] - before[1] == 5
            taus.append([float(ctx.get_tensor(B.T_TAU, l)[0]) for l in range(2, 15)])
        bits.append(taus)
        if run == 0:
            for l in range(1, 14):
                g = o.grad_p_phi(s.p[l], s.W[l], s.b[l], s.z[l], prm.nu, s.q[l - 1], s.u[l - 1], prm.rho)
                first = prm.rho + prm.nu * np.sum((s.W[l] @ g) ** 2) / np.sum(g ** 2)
                trials = int(ctx.get_tensor(B.T_TRIALS, l + 1)[0])
                assert abs(taus[-1][l - 1] / 2.0 ** (trials - 1) - first) <= 2e-4 * first, l
        ctx.destroy()
    assert bits[0] == bits[1] == bits[2]


@pytest.mark.parametrize("levels", [0, 256, 4096])
def test_column_sums_of_p_outlast_other_tensors(levels):
    """Setting W, b or z leaves p as it is: the next step sums r again and not X and every p.  (Beside the sums of an iteration, those of
    r_L: one launch for r, two for p.)  It is still the oracle's iteration."""
    inp = synth.make_inputs(synth.small("c2", 261, feat_dim=9, hidden=33, n_layers=4, quant_levels=levels))
    prm, s, _ = U.oracle_problem(inp)
    ctx = B.from_inputs(inp)
    ctx.step(3)
    ctx.profile(True)

    def summing(kind):
        if kind is not None:
            ctx.set_tensor(kind, 2, ctx.get_tensor(kind, 2) * np.float32(1 if kind == B.T_P else 0.75))
        before = ctx.profile_read()["finalize"]["launches"]
        ctx.step(1)
        return ctx.profile_read()["finalize"]["launches"] - before
    own = summing(None)
    assert [summing(k) - own for k in (B.T_W, B.T_B, B.T_Z, B.T_P)] == [1, 1, 1, 3]
    ctx.profile(False)
    ctx.set_tensor(B.T_W, 3, ctx.get_tensor(B.T_W, 3) * np.float32(1.25))
    for k, v in U.read_state(ctx).items():
        setattr(s, k, v)
    if levels:
        s.scale = [s.scale[0]] + [float(ctx.get_tensor(B.T_QSCALE, l)[0]) for l in (2, 3, 4)]
    _compare_iteration(ctx, s, prm, f"m={levels}")
    ctx.destroy()


def test_reading_q_of_one_layer_forms_that_layer_s():
    inp = synth.make_inputs(synth.small("c2", 261, feat_dim=9, hidden=33, n_layers=5, quant_levels=0))
    nu = np.float32(inp.workload.nu)
    ctx = B.from_inputs(inp)
    ctx.step(2)
    before = ctx.launches()
    q = {l: ctx.get_tensor(B.T_Q, l) for l in (3, 3, 1)}
    assert ctx.launches() - before == 2
    ctx.set_tensor(B.T_U, 2, ctx.get_tensor(B.T_U, 2))         # q may be set apart from z and u now: every layer's is stored
    assert ctx.launches() - before == 3
    for l in range(1, 5):
        z, u, got = (ctx.get_tensor(k, l) for k in (B.T_Z, B.T_U, B.T_Q))
        f = np.maximum(z, 0)
        assert (np.abs(got - (f + u / nu)) <= 4 * 2.0 ** -23 * (np.abs(f) + np.abs(u / nu))).all()
        assert l not in q or np.array_equal(q[l], got)
    ctx.destroy()


@pytest.mark.parametrize("levels,neg,step", [(0, 0, 0.0), (16, 0, 0.0), (256, 0, 0.0), (300, 0, 0.0), (22, 1, 1.0), (4096, 0, 0.0)])
def test_first_iteration_leaves_b_at_zero(levels, neg, step):
    """From the feasible start p stays as it is and every r is zero, so the mean that b takes is zero: the sums of p before the p-step and after it
    are the same bits."""
    inp = synth.make_inputs(synth.small("c2", 1033, feat_dim=9, hidden=33, n_layers=4, quant_levels=levels))
    ctx = B.from_inputs(inp, quant_neg_levels=neg, quant_step=step)
    p = [ctx.get_tensor(B.T_P, l) for l in range(1, 5)]
    ctx.step(1)
    for l in range(1, 5):
        assert np.array_equal(p[l - 1], ctx.get_tensor(B.T_P, l)), l
        assert not ctx.get_tensor(B.T_B, l).any(), l
    ctx.destroy()

"""BP and the regauge where their kernels change team width or branch: messages that are not
Hermitian (the prefix and suffix products take some of them transposed), vertices of every degree,
and batches on both sides of the width rules."""
import numpy as np
import pytest

from instances import make_instance, make_tree_instance
from oracle import gtqa_oracle as O
from paper_2409_12240_gb300 import gtqa as G

pytestmark = pytest.mark.gpu

# FP64: rounding of at most 2 chi^3 products over a trace near 1.  FP32 products: a sum of up to
# 2 * 16^3 terms of unit size in all, each off by at most a few 2^-24, so below 1e-4.
BOUND = {G.GTQA_FP64: 1e-10, G.GTQA_MIXED: 1e-4, G.GTQA_C64: 1e-4}


@pytest.mark.parametrize("precision", [G.GTQA_FP64, G.GTQA_MIXED, G.GTQA_C64])
@pytest.mark.parametrize("chi,kind", [(2, 3), (3, "tree"), (4, 3), (4, "tree"), (8, 3), (16, 3), (2, 4), (4, 4)])
def test_two_sweeps_from_messages_that_are_not_hermitian(chi, kind, precision):
    inst = make_tree_instance(9, 1) if kind == "tree" else make_instance(10, 2, d=kind)
    st = O.plus_state(inst.n, inst.edges)
    for k in range(4, 7):
        tZ, tX = O.schedule(k, 8, 0.3)
        st, _ = O.gtqa_layer(st, inst.colour, inst.J, inst.h, tZ, tX, chi, 1e-12, 200)
    rng = np.random.default_rng(7)
    msgs = {}
    for key, m0 in O.reconstructed_messages(st).items():
        noise = rng.standard_normal(m0.shape) + 1j * rng.standard_normal(m0.shape)
        m = m0 + 0.1 / m0.shape[0] * noise
        msgs[key] = m / np.trace(m)
    s = G.gtqa_create(inst.n, inst.edges, inst.J, inst.h, chi, inst.colour, G.gtqa_options_init(precision))
    try:
        C = G.gtqa_sizes(s)[2]
        Gp, Lp = O.to_padded(st, C, G.gtqa_max_degree(s))
        G.gtqa_set_state(s, Gp, Lp, O.messages_to_padded(st, msgs, C))
        it, dist, _ = G.gtqa_bp_sweep(s, 0.0, 2, 0)
        got = G.gtqa_get_state(s)[2]
    finally:
        G.gtqa_destroy(s)
    want, _, hist = O.bp(st, O.symmetric_gauge(st), msgs, 0.0, 2)
    bound = BOUND[precision]
    assert it == 2 and abs(dist - hist[-1]) < 10 * bound
    assert np.abs(got - O.messages_to_padded(st, want, C)).max() < bound


# the team widths change where a batch holds more than 4 vertices (FP64 BP at chi <= 4) or
# 512 / chi^2 edges (regauge) per SM, 152 of them: copies of n = 16 (24 edges) on both sides
@pytest.mark.parametrize("precision", [G.GTQA_FP64, G.GTQA_MIXED])
@pytest.mark.parametrize("chi,copies", [(4, 38), (4, 39), (4, 202), (4, 203), (8, 50), (8, 51), (2, 811)])
def test_instances_of_a_large_batch_follow_their_single_runs(chi, copies, precision):
    insts = [make_instance(16, 5 + i % 3) for i in range(copies)]
    args = (chi, [x.colour for x in insts], G.gtqa_options_init(precision))
    s = G.gtqa_create_batch([16] * copies, [x.edges for x in insts], [x.J for x in insts], [x.h for x in insts], *args)
    try:
        G.gtqa_anneal(s, 3, 6, 8, 0.3, 1e-12, 100)
        rho, lam = G.gtqa_marginals(s)[0], G.gtqa_get_state(s)[1]
    finally:
        G.gtqa_destroy(s)
    for i in range(3):
        x = insts[i]
        s = G.gtqa_create(x.n, x.edges, x.J, x.h, chi, x.colour, args[2])
        try:
            G.gtqa_anneal(s, 3, 6, 8, 0.3, 1e-12, 100)
            r1, l1 = G.gtqa_marginals(s)[0], G.gtqa_get_state(s)[1]
        finally:
            G.gtqa_destroy(s)
        for j in range(i, copies, 3):
            assert np.abs(rho[16 * j:16 * j + 16] - r1).max() < BOUND[precision]
            assert np.abs(lam[x.m * j:x.m * (j + 1)] - l1).max() < BOUND[precision]


# chi = 8: blocks of 512 threads from the instance sizes on at which one round of the smaller blocks no
# longer covers a kernel's items (two gates of a colour, one vertex, four edges per SM)
@pytest.mark.parametrize("precision,n,variants", [(G.GTQA_MIXED, 152, [0, 0, 0]), (G.GTQA_MIXED, 154, [0, 1, 0]),
                                                  (G.GTQA_MIXED, 1000, [1, 1, 1]), (G.GTQA_FP64, 1000, [1, 0, 1])])
def test_chi8_block_size_follows_the_instance(precision, n, variants):
    inst = make_instance(n, 4)
    out = []
    for shape in (None, [0, 0, 0]):
        s = G.gtqa_create(inst.n, inst.edges, inst.J, inst.h, 8, inst.colour, G.gtqa_options_init(precision))
        try:
            t = G.gtqa_launch_shape(s)
            assert [t[k]["variant"] for k in ("gates_kernel", "bp_kernel", "regauge_kernel")] == variants
            if shape:
                G.gtqa_set_shape(s, shape)
            G.gtqa_anneal(s, 3, 5, 8, 0.3, 1e-12, 100)
            out.append((G.gtqa_marginals(s)[0], G.gtqa_get_state(s)[1]))
        finally:
            G.gtqa_destroy(s)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])   # the same teams

"""Decompositions of the gates and the regauge where their FP32 first stage resolves least:
degenerate spectra (equal couplings, no fields), spectra graded over many orders (tiny angles),
gates of a very large or small norm, and every storage bond dimension, against the oracle."""
import numpy as np
import pytest

from instances import make_instance, random_gate_inputs
from oracle import gtqa_oracle as O
from paper_2409_12240_gb300 import gtqa as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [2, 3, 4, 8])
@pytest.mark.parametrize("couplings,dt", [("degenerate", 0.3), ("gaussian", 1e-4), ("gaussian", 0.3)])
def test_anneal_with_degenerate_and_graded_spectra(chi, couplings, dt):
    inst = make_instance(10, 3)
    J = np.ones_like(inst.J) if couplings == "degenerate" else inst.J
    h = np.zeros_like(inst.h) if couplings == "degenerate" else inst.h
    K, tol = 5, 1e-12
    for precision, bound in ((G.GTQA_FP64, 1e-10), (G.GTQA_MIXED, 1e-4)):
        s = G.gtqa_create(inst.n, inst.edges, J, h, chi, inst.colour, G.gtqa_options_init(precision))
        try:
            st = O.plus_state(inst.n, inst.edges)
            G.gtqa_anneal(s, 1, K, K, dt, tol, 100)
            for k in range(1, K + 1):
                tZ, tX = O.schedule(k, K, dt)
                st, _ = O.gtqa_layer(st, inst.colour, J, h, tZ, tX, chi, tol, 100)
            rho, _ = G.gtqa_marginals(s)
            lam = G.gtqa_get_state(s)[1]
        finally:
            G.gtqa_destroy(s)
        ref = O.to_padded(st, lam.shape[1])[1]
        assert np.abs(rho - O.reduced_density_matrices(st)).max() < bound
        assert np.abs(lam - ref).max() < bound


@pytest.mark.parametrize("chi", [2, 4, 8])
@pytest.mark.parametrize("scale", [1e-30, 1.0, 1e30])
def test_gates_of_any_norm(chi, scale):
    """A gate's scalar factor drops out of the normalised bond weights and marginals."""
    inst = make_instance(10, 1)
    edge, U, _, _ = random_gate_inputs(inst.n, inst.m, 2 * inst.m, 0, seed=4)
    s = G.gtqa_create(inst.n, inst.edges, inst.J, inst.h, chi, inst.colour)
    try:
        G.gtqa_apply_gates(s, edge, scale * U)
        G.gtqa_bp_sweep(s, 1e-12, 200)
        rho, _ = G.gtqa_marginals(s)
        lam = G.gtqa_get_state(s)[1]
    finally:
        G.gtqa_destroy(s)
    st = O.plus_state(inst.n, inst.edges)
    O.apply_gates(st, list(zip(edge.tolist(), U)), chi)
    st, _ = O.regauge(st, 1e-12, 200)
    assert np.abs(rho - O.reduced_density_matrices(st)).max() < 1e-10
    assert np.abs(lam - O.to_padded(st, lam.shape[1])[1]).max() < 1e-10

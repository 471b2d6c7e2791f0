"""The mixed mode over the range of complex64: a uniform factor of a vertex tensor drops out of the
messages, the bond weights and the marginals."""
import functools

import numpy as np
import pytest

from instances import make_instance
from oracle import gtqa_oracle as O
from paper_2409_12240_gb300 import gtqa as G

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def reference(chi, degree):
    """A state of random tensors, whose messages lie far from the warm start, and the oracle's two sweeps
    and regauge of it."""
    inst = make_instance(10, 2, d=degree)
    rng = np.random.default_rng(3)
    st = O.plus_state(inst.n, inst.edges)
    st.lam = [np.sort(rng.uniform(0.3, 1.0, chi))[::-1].copy() for _ in range(st.m)]
    for a in range(st.n):
        shape = (2,) + (chi,) * len(st.inc[a])
        g = rng.standard_normal(shape) + 1j * rng.standard_normal(shape) + 1.0
        st.Gamma[a] = g / np.linalg.norm(g)
    T, m0 = O.symmetric_gauge(st), O.reconstructed_messages(st)
    msgs, _, hist = O.bp(st, T, m0, 0.0, 2)
    assert min(np.abs(msgs[k] - m0[k]).max() for k in m0) > 1e-2
    ref = O.vidal_gauge(st, T, msgs)
    return (inst, O.to_padded(st, chi, degree), O.messages_to_padded(st, m0, chi), hist[-1],
            O.messages_to_padded(st, msgs, chi), O.to_padded(ref, chi, degree)[1], O.reduced_density_matrices(ref))


@pytest.mark.parametrize("chi,degree", [(2, 3), (4, 3), (8, 3), (16, 3), (4, 4)])
@pytest.mark.parametrize("scale", [1e-15, 1e-12, 1e-10, 1e-5, 1.0, 1e5, 1e10, 1e15])
def test_bp_and_regauge_with_scaled_vertices(chi, degree, scale):
    """The stated 1e-4 of the mixed mode on messages, bond weights and marginals."""
    inst, (Gp, Lp), m0, dist0, msgs0, lam0, rho0 = reference(chi, degree)
    s = G.gtqa_create(inst.n, inst.edges, inst.J, inst.h, chi, inst.colour, G.gtqa_options_init(G.GTQA_MIXED))
    try:
        G.gtqa_set_state(s, Gp, Lp, m0)
        G.gtqa_apply_single_qubit_gates(s, [0, 5], np.array([scale * np.eye(2)] * 2))
        it, dist, _ = G.gtqa_bp_sweep(s, 0.0, 2, G.GTQA_BP_WARM_START)
        msgs = G.gtqa_get_state(s)[2]
        G.gtqa_regauge(s)
        rho, _ = G.gtqa_marginals(s)
        lam = G.gtqa_get_state(s)[1]
    finally:
        G.gtqa_destroy(s)
    assert it == 2 and abs(dist - dist0) < 1e-4 * dist0
    assert np.abs(msgs - msgs0).max() < 1e-4
    assert np.abs(lam - lam0).max() < 1e-4
    assert np.abs(rho - rho0).max() < 1e-4

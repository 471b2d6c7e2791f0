"""Errors inside a run of the plain path are reported and end the run."""
import time

import numpy as np
import pytest

from instances import make_instance
from paper_2409_12240_gb300 import gtqa as G

pytestmark = pytest.mark.gpu

SHAPES = [(2, 4, G.GTQA_FP64), (4, 4, G.GTQA_FP64), (4, 4, G.GTQA_MIXED), (2, 3, G.GTQA_C64), (4, 3, G.GTQA_C64),
          (8, 3, G.GTQA_C64), (16, 3, G.GTQA_FP64), (16, 3, G.GTQA_MIXED), (16, 3, G.GTQA_C64)]


def plain_state(chi, degree, precision):
    inst = make_instance(10, 2, d=degree)
    s = G.gtqa_create(inst.n, inst.edges, inst.J, inst.h, chi, inst.colour, G.gtqa_options_init(precision))
    return inst, s


@pytest.mark.parametrize("call", ["bp_sweep", "anneal", "anneal_ex"])
@pytest.mark.parametrize("chi,degree,precision", SHAPES)
def test_nan_is_reported(chi, degree, precision, call):
    inst, s = plain_state(chi, degree, precision)
    try:
        G.gtqa_anneal(s, 1, 3, 8, 0.3, 1e-6, 20)
        Gam, lam, msg = G.gtqa_get_state(s)
        Gam[3].reshape(-1)[0] = np.nan
        G.gtqa_set_state(s, Gam, lam, msg)
        with pytest.raises(G.GTQAError) as err:
            if call == "bp_sweep":
                G.gtqa_trotter_layer(s, 0.5, 0.3)
                G.gtqa_bp_sweep(s, 1e-6, 20)
            elif call == "anneal":
                G.gtqa_anneal(s, 4, 6, 8, 0.3, 1e-6, 20)
            else:
                G.gtqa_anneal_ex(s, 4, 6, 8, 0.3, 1e-6, 20, G.GTQA_TROTTER_SYMMETRIC)
        assert err.value.code == G.GTQA_ERR_NUMERIC
    finally:
        G.gtqa_destroy(s)


@pytest.mark.parametrize("chi,degree,precision", SHAPES)
def test_layers_after_a_barrier_that_gave_up_do_not_run(chi, degree, precision):
    """One barrier waits for an arrival that does not come and gives up; forty layers take no longer
    over it than one."""
    took = {}
    for layers in (1, 40):
        _, s = plain_state(chi, degree, precision)
        try:
            G.gtqa_debug_barrier(s, 100000, 1)
            t = time.perf_counter()
            with pytest.raises(G.GTQAError) as err:
                G.gtqa_anneal(s, 1, layers, 40, 0.3, 1e-6, 20)
            took[layers] = time.perf_counter() - t
            assert err.value.code == G.GTQA_ERR_TIMEOUT
        finally:
            G.gtqa_destroy(s)
    assert took[40] < 5 * took[1] + 0.1

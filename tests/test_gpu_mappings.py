"""Mappings and launch lengths that are set by hand, and the planned one beside them, against the oracle
bit for bit."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1605_03607_gb300 as pkg
    from paper_1605_03607_gb300 import build as b
    b.build()
    pkg.load()
    return pkg


def same_state(st, ref):
    for k in ("spins", "E", "best", "first", "macc", "xacc"):
        assert np.array_equal(st[k], getattr(ref, k)), k


@pytest.mark.parametrize("L", [7, 14])
def test_launch_length_of_a_planned_handle(P, L):
    J, betas = W.random_couplers(L, 5, L), W.beta_ladder(12, 0.1, 3.0)
    ref = oracle.PTState(L, J, betas, 3, 5, L)
    ref.sweeps(20, 2)
    with P.PTHandle(L, J, betas, 3, 5, L) as h:
        h.set_schedule(0, 0, 7)
        assert h.schedule()[2] == 7
        h.sweep(20, 2)
        same_state(h.state(), ref)

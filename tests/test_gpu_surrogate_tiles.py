"""The surrogate's kernels where their tiles have edges: 128 nodes or 128 edges per tile, across
graph borders, against batch sizes and lattice sides that leave every remainder, and one to
eight layers (the last one updates no edges).  Two properties that hold for any tiling:

* a graph's prediction does not depend on the graphs beside it, bit for bit (its rows meet the
  same operations in the same order in every tile);
* with 32 graphs the gradient is the mean of the graphs' own gradients.  Dividing by 32 commutes
  with every rounding to BF16, so the two differ only by the order of FP32 sums of at most
  n = 32 * 2 * 1232 rows: sqrt(n) 2^-24 = 2e-5 of the largest partial sum; 1e-4 of a tensor's
  largest entry is allowed.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1605_03607_gb300 as pkg
    from paper_1605_03607_gb300 import build as b
    b.build()
    pkg.load()
    return pkg


def _case(L, B, layers, seed):
    rng = np.random.default_rng(seed)
    J = rng.choice([-3, -2, -1, 1, 2, 3], size=(B, W.chimera_n_edges(L))).astype(np.int8)
    th = W.surrogate_init_params(seed, layers=layers)
    return J, (th + 0.02 * rng.standard_normal(len(th))).astype(np.float32), rng.uniform(1.5, 4.0, B)


@pytest.mark.parametrize("L,layers", [(1, 4), (2, 1), (3, 4), (5, 2), (7, 4), (16, 8)])
def test_predictions_do_not_depend_on_the_batch(P, L, layers):
    J, th, _ = _case(L, 45 if L < 16 else 5, layers, L)
    with P.Surrogate(layers=layers) as m:
        m.set_params(th)
        y = m.forward(L, J)
        for a, b in ((0, 1), (0, 2), (1, 4), (0, 20), (3, 24), (0, 44)):
            if b <= len(J):
                assert np.array_equal(m.forward(L, J[a:b]), y[a:b]), (a, b)


@pytest.mark.parametrize("L,layers", [(1, 4), (3, 1), (3, 4), (4, 2), (7, 4)])
def test_gradient_is_the_mean_of_single_graphs(P, L, layers):
    B = 32
    J, th, t = _case(L, B, layers, 40 + L)
    with P.Surrogate(layers=layers) as m:
        m.set_params(th)
        loss, g = m.grad(L, J, t)
        each = [m.grad(L, J[b:b + 1], t[b:b + 1]) for b in range(B)]
    assert abs(loss - np.mean([e[0] for e in each])) <= 1e-6 * abs(loss)
    want = np.mean([e[1].astype(np.float64) for e in each], axis=0)
    o = 0
    for name, n, _ in W.surrogate_param_sizes(layers=layers):
        a, b = g[o:o + n], want[o:o + n]
        o += n
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max(), name

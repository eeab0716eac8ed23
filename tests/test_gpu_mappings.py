"""Mappings and launch lengths that are set by hand, and the planned one beside them, against the oracle
bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


CELL_MAJOR = [
    # L, NT, R, sweeps, exchange_every: the default cell-major schedule, also where a plan would take other lanes
    (4, 16, 8, 200, 1),
    (8, 32, 4, 60, 1),
    (12, 24, 2, 20, 1),
    (16, 48, 2, 8, 1),
    (1, 4, 3, 300, 1),                          # a warp spans many slots
    (2, 6, 3, 300, 1),
    (3, 5, 2, 100, 2),
    (5, 8, 2, 100, 1),
    (4, 2, 4, 150, 1),
    (4, 64, 2, 40, 1),                          # most slots
    (4, 33, 3, 90, 1),                          # two slots per exchange lane
    (16, 4, 3, 20, 1),                          # few temperatures: also the planned mapping
]


@pytest.mark.parametrize("walk", [False, True])
@pytest.mark.parametrize("L,NT,R,n,x", CELL_MAJOR)
def test_cell_major_bit_exact(P, L, NT, R, n, x, walk):
    J, betas = W.random_couplers(L, 11 + L, NT), W.beta_ladder(NT, 0.1, 3.0)
    ref = oracle.PTState(L, J, betas, R, 11 + L, NT, walk=walk)
    with P.PTHandle(L, J, betas, R, 11 + L, NT) as h:
        h.set_mapping(0)
        assert h.launch_shape()["mapping"] == "cell-major"
        h.set_walk_stats(walk)
        for part in (n // 2, n - n // 2):
            h.sweep(part, x)
            ref.sweeps(part, x)
            h.exchange()
            ref.exchange()
        same_state(h.state(), ref)
        if walk:
            hot, trips, passes = h.walk_stats()
            assert passes == ref.n_passes and np.array_equal(hot, ref.hot) and np.array_equal(trips, ref.trips)


def test_narrow_ladder_cell_major(P):
    """Exchange tables of about 15,000 entries a pair: the critical gaps' float estimate at its largest error."""
    J, betas = W.random_couplers(2, 31, 5), W.beta_ladder(64, 0.30, 0.35)
    ref = oracle.PTState(2, J, betas, 4, 31, 5)
    ref.sweeps(300, 1)
    with P.PTHandle(2, J, betas, 4, 31, 5) as h:
        h.set_mapping(0)
        h.sweep(300, 1)
        same_state(h.state(), ref)
    assert ref.xacc.sum() > 0


@pytest.mark.parametrize("L,NT,R,mapping", [(4, 16, 8, "replica-lane"), (8, 32, 3, "replica-lane"), (7, 30, 7, "replica-lane"),
                                            (16, 4, 3, "cell-major"), (16, 8, 1, "cell-major"), (12, 5, 2, "cell-major")])
def test_planned_mapping_of_a_size(P, L, NT, R, mapping):
    """The sizes of the planned mapping's tests take the mapping that they are there for."""
    with P.PTHandle(L, W.random_couplers(L, 1, 0), W.beta_ladder(NT, 0.1, 3.0), R, 1, 0) as h:
        assert h.launch_shape()["mapping"] == mapping


@pytest.mark.parametrize("L,NT,R", [(2, 1, 9), (2, 13, 1000), (2, 33, 5), (2, 64, 130), (1, 5, 600), (3, 32, 70)])
@pytest.mark.parametrize("spl", [1, 4])
def test_short_launches_of_small_lattices(P, L, NT, R, spl):
    """Every launch stages and writes back the state, many runs a CTA."""
    J, betas = W.random_couplers(L, 4, NT), W.beta_ladder(NT, 0.1, 3.0) if NT > 1 else np.array([1.0])
    ref = oracle.PTState(L, J, betas, R, 4, NT)
    ref.sweeps(9, 1)
    with P.PTHandle(L, J, betas, R, 4, NT) as h:
        h.set_schedule(0, 0, spl)
        h.sweep(9, 1)
        st = h.state()
    for k in ("spins", "E", "best", "first", "macc") + (("xacc",) if NT > 1 else ()):
        assert np.array_equal(st[k], getattr(ref, k)), k


@pytest.mark.parametrize("L,NT,R", [(4, 2, 3), (8, 32, 70), (7, 33, 5), (12, 24, 16), (16, 64, 2), (2, 40, 300)])
def test_exchanges_alone(P, L, NT, R):
    """Exchange passes of their own, one after another and between sweeps, with the walk tracked."""
    J, betas = W.random_couplers(L, 6, NT), W.beta_ladder(NT, 0.1, 3.0)
    ref = oracle.PTState(L, J, betas, R, 6, NT, walk=True)
    with P.PTHandle(L, J, betas, R, 6, NT) as h:
        h.set_walk_stats(True)
        for n in (0, 2, 1):
            h.sweep(n, 0)
            ref.sweeps(n, 0)
            for _ in range(3):
                h.exchange()
                ref.exchange()
        hot, trips, passes = h.walk_stats()
        st = h.state()
        same_state(st, ref)
        assert np.array_equal(st["E"], ref.full_energies())
    assert passes == ref.n_passes and np.array_equal(hot, ref.hot) and np.array_equal(trips, ref.trips)


@pytest.mark.parametrize("L,NT,R,k", [(2, 17, 25, 24), (3, 7, 100, 24), (6, 17, 25, 24), (8, 7, 256, 16)])
def test_candidates_share_ctas(P, L, NT, R, k):
    """Candidates whose run counts do not divide into whole CTAs: some CTA holds runs of two."""
    J = np.stack([W.random_couplers(L, 5, j) for j in range(k)])
    betas = W.beta_ladder(NT, 0.1, 3.0)
    with P.PTHandle(L, J[0], betas, R, 5, 0) as h:
        assert h.launch_shape(k)["shared_ctas"] > 0
        out = h.tts_eval_many(J, np.arange(k) + 3, 3)
    for j in range(k):
        assert (out["tts"][j], out["n_hit"][j], out["target"][j]) == oracle.tts_eval(L, J[j], betas, R, 5, j + 3, 3, 1, 1), j


def test_batch_reports_what_it_runs(P):
    inst = [dict(L=L, J=W.random_couplers(L, 2, i), betas=W.beta_ladder(NT, 0.1, 3.0), uid=i)
            for i, (L, NT) in enumerate([(4, 24), (4, 30), (16, 4)])]
    with P.PTBatch(inst, 3, 2) as b:
        assert b.launch_shape(4)["mapping"] == "replica-lane" and b.launch_shape(16)["mapping"] == "cell-major"
        b.set_mapping(4, 4, 30, 1)
        s = b.launch_shape(4)
        assert (s["mapping"], s["team"], s["runs_per_cta"], s["threads"]) == ("slot-major", 4, 1, 128)


DEBUG_SCRIPT = r'''
import sys
sys.path.insert(0, ROOT)
import numpy as np
from paper_1605_03607_gb300 import build as b
b.build(debug=True)
import paper_1605_03607_gb300 as P
import oracle
import workloads as W
assert P.debug_enabled(), "not the debug build"
for L, NT, R, set_it in ((4, 8, 4, True), (8, 32, 3, True), (16, 4, 3, False), (3, 40, 5, True)):
    J, betas = W.random_couplers(L, 20160519, 0), W.beta_ladder(NT, 0.1, 3.0)
    ref = oracle.PTState(L, J, betas, R, 20160519, 1)
    ref.sweeps(40, 1)
    ref.exchange()
    for walk in (False, True):
        with P.PTHandle(L, J, betas, R, 20160519, 1) as h:
            if set_it:
                h.set_mapping(0)
            assert h.launch_shape()["mapping"] == "cell-major"
            h.set_walk_stats(walk)
            h.sweep(40, 1)
            h.exchange()
            st = h.state()
        assert np.array_equal(st["spins"], ref.spins) and np.array_equal(st["E"], ref.E)
        assert np.array_equal(st["best"], ref.best) and np.array_equal(st["first"], ref.first)
code = P.debug_status()
assert code == 0, f"bounds check {code} failed"
print("debug build: no failed bounds check")
'''


def test_debug_build_runs_clean_cell_major():
    env = dict(os.environ, PT_GB300_DEBUG="1")
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + DEBUG_SCRIPT], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]
    assert "no failed bounds check" in r.stdout
    assert "PT_DEBUG" not in r.stderr

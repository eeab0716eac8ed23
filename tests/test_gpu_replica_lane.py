"""The planned (replica-lane) mapping against the oracle, bit for bit, at the sizes where its
layout has edges: odd sides (cell pairs, a last single cell), runs that share columns of 32
replicas, partly filled columns and groups, two-word exchange masks, the longest threshold
tables, and standalone exchange passes between split sweeps."""
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


SHAPES = [
    # L, NT, R, sweeps, exchange_every
    (1, 1, 70, 40, 1),          # one cell, one temperature
    (2, 3, 1024, 12, 1),        # two runs a column
    (3, 5, 1000, 9, 2),         # odd side, four runs a column, fewer warps than cell pairs
    (4, 6, 1023, 10, 1),        # the last group short of runs
    (4, 32, 5, 60, 1),          # columns exactly full
    (4, 33, 5, 60, 1),          # one replica in the second column
    (4, 48, 1024, 3, 1),        # two runs on three columns
    (4, 64, 3, 60, 3),
    (5, 20, 700, 4, 1),         # odd side, three runs on two columns
    (6, 40, 603, 3, 1),         # four runs on five columns
    (7, 30, 7, 30, 10),
    (9, 64, 2, 12, 1),
    (10, 36, 160, 2, 1),
    (11, 17, 3, 12, 1),
    (13, 40, 2, 8, 1),
    (14, 33, 2, 8, 1),
    (15, 9, 2, 8, 1),
    (16, 64, 2, 6, 1),
]


@pytest.mark.parametrize("L,NT,R,n,x", SHAPES)
def test_planned_mapping_bit_exact(P, L, NT, R, n, x):
    J = W.random_couplers(L, 31 + L, NT)
    betas = W.beta_ladder(NT, 0.1, 3.0)
    ref = oracle.PTState(L, J, betas, R, 31 + L, NT)
    with P.PTHandle(L, J, betas, R, 31 + L, NT) as h:
        for part in (n // 3, n - n // 3):
            h.sweep(part, x)
            ref.sweeps(part, x)
            h.exchange()
            ref.exchange()
        st = h.state()
    for k in ("spins", "E", "best", "first", "macc") + (("xacc",) if NT > 1 else ()):
        assert np.array_equal(st[k], getattr(ref, k)), k
    assert np.array_equal(st["E"], ref.full_energies())


@pytest.mark.parametrize("L,NT,R,walk", [(16, 4, 3, False), (16, 8, 1, True), (12, 5, 2, False), (8, 2, 1, False), (6, 1, 4, False),
                                         (12, 2, 200, False)])
def test_planned_few_temperatures(P, L, NT, R, walk):
    """Few replicas on a large lattice: a plan may take a lane per cell, with the same bytes, also for a single
    exchange, for candidates of fewer runs (a doubling budget) and in the evaluation without allocation."""
    J = W.random_couplers(L, 3, NT)
    betas = W.beta_ladder(NT, 0.1, 3.0) if NT > 1 else np.array([1.0])
    ref = oracle.PTState(L, J, betas, R, 3, NT)
    with P.PTHandle(L, J, betas, R, 3, NT) as h:
        if walk:
            h.set_walk_stats(True)
        h.sweep(5, 1)
        h.exchange()
        h.sweep(4, 2)
        ref.sweeps(5, 1)
        ref.exchange()
        ref.sweeps(4, 2)
        st = h.state()
        for k in ("spins", "E", "best", "first", "macc") + (("xacc",) if NT > 1 else ()):
            assert np.array_equal(st[k], getattr(ref, k)), k
        out = h.tts_eval_many(np.stack([J, J]), [1, 2], 2, max_sweeps=4)
    for i in range(2):
        assert (out["tts"][i], out["n_hit"][i], out["target"][i]) == tuple(
            oracle.tts_eval_doubling(L, J, betas, R, 3, i + 1, 2, 4, 1)[:3])


@pytest.mark.parametrize("L,NT,R,k", [(4, 24, 64, 16), (6, 20, 24, 3)])
def test_planned_groups_of_candidates(P, L, NT, R, k):
    """Several groups per CTA and several CTAs per instance, every candidate with its own couplers."""
    betas = W.beta_ladder(NT, 0.1, 3.0)
    Js = np.stack([W.random_couplers(L, 5, j) for j in range(k)])
    with P.PTHandle(L, Js[0], betas, R, 5, 0) as h:
        out = h.tts_eval_many(Js, np.arange(k) + 3, 6, 2)
    for j in range(k):
        want = oracle.tts_eval(L, Js[j], betas, R, 5, j + 3, 6, 2, 1)
        assert (out["tts"][j], out["n_hit"][j], out["target"][j]) == want, j


@pytest.mark.parametrize("L,NT,R,k", [(2, 17, 25, 24), (3, 7, 100, 24), (6, 17, 25, 24), (8, 7, 256, 16)])
@pytest.mark.parametrize("adaptive", [False, True])
def test_planned_ctas_of_two_instances(P, L, NT, R, k, adaptive):
    """Run counts that do not divide into whole CTAs: the last runs of one candidate share a CTA
    with the first of the next.  With a doubling budget the candidates of a launch are no
    longer consecutive and the shape changes from level to level."""
    betas = W.beta_ladder(NT, 0.1, 3.0)
    Js = np.stack([W.random_couplers(L, 5, j) for j in range(k)])
    uids = np.arange(k) + 3
    with P.PTHandle(L, Js[0], betas, R, 5, 0) as h:
        out = h.tts_eval_many(Js, uids, 1 if adaptive else 4, 1, max_sweeps=8 if adaptive else 0)
    for j in range(k):
        if adaptive:
            want = oracle.tts_eval_doubling(L, Js[j], betas, R, 5, j + 3, 1, 8, 1)
            assert (out["tts"][j], out["n_hit"][j], out["target"][j]) == tuple(want[:3]), j
        else:
            want = oracle.tts_eval(L, Js[j], betas, R, 5, j + 3, 4, 1, 1)
            assert (out["tts"][j], out["n_hit"][j], out["target"][j]) == want, j


@pytest.mark.parametrize("L,kmax", [(1, 127), (2, 127), (3, 64)])
def test_planned_longest_tables(P, L, kmax):
    """Local fields up to the largest allowed: the byte 127 + k of a field spans 0..254."""
    rng = np.random.default_rng(L)
    J = rng.integers(-127, 128, size=W.chimera_n_edges(L)).astype(np.int64)
    while oracle.coupler_kmax(L, J.astype(np.int8)) > kmax:
        J = np.sign(J) * (np.abs(J) * 9 // 10)
    e = 0                                        # raise one spin's sum to exactly kmax
    while oracle.coupler_kmax(L, J.astype(np.int8)) < kmax and e < len(J):
        J[e] += 1 if J[e] >= 0 else -1
        if oracle.coupler_kmax(L, J.astype(np.int8)) > kmax or abs(J[e]) > 127:
            J[e] -= 1 if J[e] > 0 else -1
            e += 1
    J = J.astype(np.int8)
    assert oracle.coupler_kmax(L, J) == kmax
    betas = W.beta_ladder(12, 0.004, 0.3)
    ref = oracle.PTState(L, J, betas, 5, 9, 1)
    ref.sweeps(150, 1)
    with P.PTHandle(L, J, betas, 5, 9, 1) as h:
        h.sweep(150, 1)
        st = h.state()
    for k in ("spins", "E", "best", "first", "macc", "xacc"):
        assert np.array_equal(st[k], getattr(ref, k)), k


def test_planned_batch_of_uneven_instances(P):
    """One CTA size for instances of 24 to 48 temperatures: groups of different column counts,
    CTAs with idle warps, last groups short of runs."""
    R, seed = 9, 77
    inst = [dict(L=L, J=W.random_couplers(L, seed, i), betas=W.beta_ladder(NT, 0.1, 3.0), uid=i)
            for i, (L, NT) in enumerate([(4, 24), (4, 33), (4, 48), (3, 30), (3, 40), (6, 36), (4, 1)])]
    with P.PTBatch(inst, R, seed) as b:
        b.run(7, 1)
        b.run(12, 2)
        for i, x in enumerate(inst):
            st = b.state(i)
            ref = oracle.PTState(x["L"], x["J"], x["betas"], R, seed, i)
            ref.sweeps(7, 1)
            ref.sweeps(12, 2)
            for k in ("spins", "E", "best", "first", "macc") + (("xacc",) if len(x["betas"]) > 1 else ()):
                assert np.array_equal(st[k], getattr(ref, k)), (i, k)


@pytest.mark.parametrize("n", [2, 40])
def test_planned_batch_of_few_temperatures(P, n):
    """Batches whose groups have up to 10 temperatures: cell-major groups for few CTAs on a large lattice."""
    R, seed = 2, 78
    inst = [dict(L=L, J=W.random_couplers(L, seed, i), betas=W.beta_ladder(NT, 0.1, 3.0), uid=i)
            for i, (L, NT) in enumerate([(16, 4), (12, 5), (4, 8)] * n)][:n + 1]
    with P.PTBatch(inst, R, seed) as b:
        b.run(6, 1)
        b.run(5, 2)
        for i, x in enumerate(inst):
            st = b.state(i)
            ref = oracle.PTState(x["L"], x["J"], x["betas"], R, seed, i)
            ref.sweeps(6, 1)
            ref.sweeps(5, 2)
            for k in ("spins", "E", "best", "first", "macc", "xacc"):
                assert np.array_equal(st[k], getattr(ref, k)), (i, k)

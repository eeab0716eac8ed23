"""The handle runtime's launch lists and copies on error paths, on the CPU (tests/host_runtime.py)."""
import threading

import numpy as np
import pytest

import host_runtime
import workloads as W


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    lib = host_runtime.build(tmp_path_factory.mktemp("host_runtime"))
    if lib is None:
        pytest.skip("no host compiler or CUDA headers")
    return lib


@pytest.fixture
def rt(host_lib, monkeypatch):
    from paper_1605_03607_gb300 import _lib
    monkeypatch.setattr(_lib, "_lib", host_lib)
    host_lib.host_fail_launches(0, 0)
    host_lib.host_fail_allocs(0, 0)
    host_lib.host_fastest(0, -1)
    before = host_lib.host_overruns()
    yield host_lib
    host_lib.host_fail_launches(0, 0)
    host_lib.host_fail_allocs(0, 0)
    assert host_lib.host_overruns() == before


def handle(L, NT, R):
    import paper_1605_03607_gb300 as P
    return P.PTHandle(L, W.random_couplers(L, 3, 0), W.beta_ladder(NT, 0.1, 3.0), R, 3, 0)


def evaluate(rt, h, k):
    """Candidates, and the handle's own runs under a doubling budget: every run in the launches once."""
    J = np.stack([h.couplers()] * k)
    h.tts_eval_many(J, np.arange(k), 4)
    assert rt.host_last_launch_ok(k, h.R)
    h.tts_eval_many(J[:1], np.arange(1), 4, max_sweeps=8)
    assert rt.host_last_launch_ok(1, h.R)
    h.tts_eval_doubling(1, 4, 8)
    assert rt.host_last_launch_ok(1, h.R)


@pytest.mark.parametrize("L,NT,R,k", [(16, 48, 32, 4), (8, 32, 64, 1), (7, 30, 100, 3), (4, 6, 40, 2)])
@pytest.mark.parametrize("what", ["launches", "allocs"])
def test_failed_autotune_leaves_launchable_lists(rt, L, NT, R, k, what):
    """A tuning run that fails at its n-th launch, or from its n-th allocation on, for every n."""
    import paper_1605_03607_gb300 as P
    with handle(L, NT, R) as h:
        rt.host_fail_launches(0, 0)
        rt.host_fail_allocs(0, 0)
        h.autotune(k, 2)
        total = getattr(rt, "host_" + what)()
    assert total > 3
    for n in range(1, total + 1):
        with handle(L, NT, R) as h:
            getattr(rt, "host_fail_" + what)(n, total + 1000)
            with pytest.raises(P.PTError):
                h.autotune(k, 2)
            getattr(rt, "host_fail_" + what)(0, 0)
            evaluate(rt, h, k)


@pytest.mark.parametrize("L,NT,R,k", [(16, 48, 32, 4), (8, 32, 64, 2)])
def test_failed_mapping_change_leaves_launchable_lists(rt, L, NT, R, k):
    """A change of mapping that runs out of memory, with the way back failing too or not."""
    import paper_1605_03607_gb300 as P
    for n in range(1, 9):
        for last in (n, 1000):
            with handle(L, NT, R) as h:
                evaluate(rt, h, k)
                rt.host_fail_allocs(n, last)
                try:
                    h.set_mapping(4, NT, 2 if L == 8 else 1)
                    failed = False
                except P.PTError:
                    failed = True
                rt.host_fail_allocs(0, 0)
                assert failed == (n <= 4)        # two groups, two lists each
                evaluate(rt, h, k)


@pytest.mark.parametrize("L", [4, 7, 11, 14, 15])
def test_launch_length_of_a_planned_handle(rt, L):
    """A new launch length keeps the plan, also where the set mappings' default does not fit a CTA."""
    with handle(L, 20, 6) as h:
        rt.host_fail_launches(0, 0)
        h.sweep(20, 1)
        assert rt.host_launches() == 1
        block = rt.host_last_block()
        h.set_schedule(0, 0, 7)
        assert h.schedule()[2] == 7
        rt.host_fail_launches(0, 0)
        h.sweep(20, 1)
        assert rt.host_launches() == 3 and rt.host_last_team() < 0 and rt.host_last_block() == block


@pytest.mark.parametrize("L,NT,team,block", [(16, 55, 0, 1024), (11, 51, 2, 408)])
def test_autotune_keeps_a_schedule_that_the_walk_counters_fit(rt, L, NT, team, block):
    """The fastest trial fits a CTA without the main runs' walk counters and not with them."""
    with handle(L, NT, 4) as h:
        h.set_walk_stats(True)
        rt.host_fastest(team, block)
        h.autotune(2, 2)
        h.sweep(3, 1)
        assert rt.host_last_launch_ok(1, 4)
        evaluate(rt, h, 2)


@pytest.mark.parametrize("L,NT,R", [(2, 64, 1024), (4, 30, 700), (4, 16, 8), (8, 32, 64), (2, 1, 3)])
def test_state_downloads_what_is_asked_for(rt, L, NT, R):
    """Records too large for the staging: only the arrays asked for are copied, each once."""
    from paper_1605_03607_gb300._lib import _ptr
    N, x, r = 8 * L * L, np.arange(R * NT), np.arange(R)
    with handle(L, NT, R) as h:
        s = np.where(np.random.default_rng(1).random((R, NT, N)) < 0.5, -1, 1).astype(np.int8)
        h.set_spins(s)
        want = dict(spins=s[:, ::-1].copy(), E=(7 * x + 3).astype(np.int32),
                    perm=np.tile(np.arange(NT)[::-1], R).astype(np.uint8), best=(-r).astype(np.int32),
                    first=(r + 1).astype(np.int32), macc=(11 * x).astype(np.uint64),
                    xacc=(13 * np.arange(R * (NT - 1))).astype(np.uint64))
        large = sum(a.nbytes for k, a in want.items() if k != "spins") > 256 * 1024
        for names in (tuple(want), ("E",), ("spins",), ("spins", "perm"), ("best", "xacc")):
            out = {k: np.full(want[k].shape, 99, want[k].dtype) for k in names}
            rt.host_downloaded()
            assert rt.pt_get_state(h.h, *(_ptr(out.get(k)) for k in want), None) == 0
            got = rt.host_downloaded()
            if large:
                assert got == sum(want[k].nbytes for k in set(names) | ({"perm"} if "spins" in names else set())), names
            for k in names:
                assert np.array_equal(out[k], want[k]), k


def test_state_read_by_two_threads(rt):
    """Two threads that read one handle, one everything and one the energies: neither sees the other's copy."""
    from paper_1605_03607_gb300._lib import _ptr
    L, NT, R = 4, 16, 8
    with handle(L, NT, R) as h:
        s = np.where(np.random.default_rng(2).random((R, NT, 8 * L * L)) < 0.5, -1, 1).astype(np.int8)
        h.set_spins(s)
        want = h.state()
        wrong = []
        rt.host_wait(300)

        def everything():
            for _ in range(60):
                st = h.state()
                if any(not np.array_equal(st[k], want[k]) for k in want):
                    wrong.append("state")

        def energies():
            for _ in range(60):
                E = np.zeros((R, NT), np.int32)
                rt.pt_get_state(h.h, None, _ptr(E), None, None, None, None, None, None)
                if not np.array_equal(E, want["E"]):
                    wrong.append("E")

        threads = [threading.Thread(target=f) for f in (everything, energies)]
        for x in threads:
            x.start()
        for x in threads:
            x.join()
        rt.host_wait(0)
        assert not wrong


SHAPES = [
    # L, NT, R, candidates, mapping of the handle's runs, CTAs of two candidates
    (8, 32, 64, 16, "replica-lane", True),
    (4, 16, 8, 4, "replica-lane", False),
    (2, 17, 25, 24, "replica-lane", True),
    (3, 7, 100, 24, "replica-lane", True),
    (6, 17, 25, 24, "replica-lane", True),
    (8, 7, 256, 16, "replica-lane", True),
    (16, 4, 3, 1, "cell-major", False),
    (16, 8, 1, 2, "cell-major", False),
    (12, 5, 2, 2, "cell-major", False),
    (12, 2, 200, 2, "cell-major", False),
    (14, 40, 3, 2, "replica-lane", False),
]


@pytest.mark.parametrize("L,NT,R,k,mapping,shared", SHAPES)
def test_launch_shape_is_what_is_launched(rt, L, NT, R, k, mapping, shared):
    with handle(L, NT, R) as h:
        s = h.launch_shape()
        h.sweep(3, 1)
        assert s["mapping"] == mapping and rt.host_last_launch_ok(1, R)
        assert (rt.host_last_team(), rt.host_last_block(), rt.host_last_ctas()) == (s["team"], s["threads"], s["ctas"])
        s = h.launch_shape(k)
        h.tts_eval_many(np.stack([h.couplers()] * k), np.arange(k), 4)
        assert rt.host_last_launch_ok(k, R) and (s["shared_ctas"] > 0) == shared
        assert (rt.host_last_team(), rt.host_last_block(), rt.host_last_ctas()) == (s["team"], s["threads"], s["ctas"])
        if L in (4, 8, 12, 16):
            for m in ((0, 1 if L == 16 else 2, 1), (4, max(NT, 8), 1)):
                h.set_mapping(*m)
                s = h.launch_shape(k)
                assert s["mapping"] == ("slot-major" if m[0] else "cell-major")
                assert (s["team"], s["slot_parallel"], s["runs_per_cta"], s["ctas"]) == (*m, k * R)


def test_planned_lists_cover_every_run_once(rt):
    """Sizes over the whole range, with the walk tracked or not, short and long threshold tables: the runs' and the
    candidates' launches hold every run once, in CTAs that fit."""
    rng = np.random.default_rng(7)
    for _ in range(150):
        L, NT, k = int(rng.integers(1, 17)), int(rng.integers(1, 65)), int(rng.integers(1, 17))
        R = min(int(np.exp(rng.uniform(0, np.log(1025)))), 1024, max(1, 20_000_000 // (8 * L * L * NT * k)))
        with handle(L, NT, R) as h:
            if rng.random() < 0.3:
                h.set_walk_stats(True)
            h.sweep(1, 1)
            assert rt.host_last_launch_ok(1, R), (L, NT, R)
            J = np.stack([h.couplers()] * k)
            if rng.random() < 0.3 and L < 15:
                J[0, :4] = 28
            h.tts_eval_many(J, np.arange(k), 4)
            assert rt.host_last_launch_ok(k, R), (L, NT, R, k)
            h.sweep(1, 1)
            assert rt.host_last_launch_ok(1, R), (L, NT, R)

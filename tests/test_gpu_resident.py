"""Whole solves in one launch (the lattice in a cluster's shared memory) against one sweep per launch:
identical populations bit for bit at the edges of its shapes (blocks of one row, a last block with
fewer rows, one to three nodes per thread, lattices one column wide), for every wall kind, with
wells, dense sources and a mid-solve rebase, and the same stopping sweep as the host's rule."""
import time

import numpy as np
import pytest

import workloads as W
from _problems import uniform

pytestmark = pytest.mark.gpu

SHAPES = [(1, 7), (5, 3), (31, 30), (64, 64), (97, 70), (300, 9), (128, 128), (131, 127), (7, 500)]
WALLS = {"periodic": (0, 0, 0, 0), "noflux": (1, 1, 1, 1), "dirichlet": (2, 2, 2, 2),
         "mixed": (0, 0, 2, 1), "mixed2": (1, 2, 0, 0)}


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_07554_gb300 import build
    build.build()
    import paper_1808_07554_gb300 as pkg
    pkg.load_library()


def _problem(nx, ny, walls):
    rng = np.random.default_rng(nx * 1000 + ny)
    dense = (nx + ny) % 2 == 0
    wells = [(0, 0, 1e-3, 0), (nx - 1, ny - 1, 1e-3, 1), (nx // 2, ny // 3, 2e-3, 0)]
    return rng, uniform(nx, ny, bc=WALLS[walls], K=np.exp(rng.standard_normal((ny, nx))),
                        S0=0.2 + 0.5 * rng.random((ny, nx)),
                        Fp=rng.standard_normal((ny, nx)) if dense else None, wells=wells,
                        P_b=[rng.random(2 * (ny if s < 2 else nx) + 1) for s in range(4)],
                        S_b=[np.full(2 * (ny if s < 2 else nx) + 1, 0.3) for s in range(4)])


@pytest.mark.parametrize("walls", list(WALLS))
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_resident_equals_single_sweeps(nx, ny, walls):
    import paper_1808_07554_gb300 as pkg
    bc = WALLS[walls]
    if (nx < 3 and 2 in bc[:2]) or (ny < 3 and 2 in bc[2:]):
        pytest.skip("Dirichlet sides need three nodes")
    rng, prob = _problem(nx, ny, walls)
    state = None
    for every, cap in ((2, 2), (2, 6), (8, 48), (8, 1040)):   # 1040: a rebase after sweep 1024
        kw = dict(init_replay=0, tol=0.0, max_sub_iters=cap, check_every=every)
        one = pkg.Solver.from_problem(prob, fuse_sweeps=1, **kw)
        res = pkg.Solver.from_problem(prob, **kw)
        assert res.fused_form() == pkg.FUSED_RESIDENT
        if state is None:
            state = one.get_state()
            state[:8] = 0.01 * rng.standard_normal(state[:8].shape)
            state[19] = rng.standard_normal(state[19].shape)
        one.set_state(state)
        res.set_state(state)
        s1, s2 = one.step(2), res.step(2)
        for t in s1[1] + s2[1]:                # the rule r <= 0: a few nodes may reach it
            assert t.sub_iters == cap or t.residual == 0.0
        if all(t.sub_iters == cap for t in s1[1] + s2[1]):
            assert np.array_equal(one.get_state(), res.get_state()), (nx, ny, walls, every, cap)
            for x, y in zip(s1[1], s2[1]):
                assert y.residual == pytest.approx(x.residual, rel=1e-3, abs=1e-9)
        else:
            assert nx * ny < 16 and cap > 48
        one.close()
        res.close()


@pytest.mark.parametrize("name", ["five_spot", "manufactured", "example2"])
def test_resident_stops_where_single_sweeps_do(name):
    """To a tolerance: the counts agree up to one check period (the residual's sums are grouped
    differently), and so do the fields; long solves cross several rebases."""
    import paper_1808_07554_gb300 as pkg
    prob = {"five_spot": lambda: W.quarter_five_spot(96, seed=3, corr_len=8.0),
            "manufactured": lambda: W.manufactured_periodic(64),
            "example2": lambda: W.example2(48)}[name]()
    one = pkg.Solver.from_problem(prob, fuse_sweeps=1, tol=1e-7)
    res = pkg.Solver.from_problem(prob, tol=1e-7)
    assert res.fused_form() == pkg.FUSED_RESIDENT
    assert abs(one.init_stats.sub_iters - res.init_stats.sub_iters) <= 8
    for _ in range(3):
        a, b = one.step(1)[1][0], res.step(1)[1][0]
        assert abs(a.sub_iters - b.sub_iters) <= 8 and b.residual <= 1e-7
    Pa, Sa = one.fields(mean_free_P=True)
    Pb, Sb = res.fields(mean_free_P=True)
    # one more check period moves P by at most 8 sweeps' increments of 1e-7 each, three solves
    assert W.rel_l2(Pb, Pa) <= 8 * 4 * 1e-7 * 2 and W.rel_l2(Sb, Sa) <= 1e-6
    one.close()
    res.close()


@pytest.mark.parametrize("nx,ny", [(5, 3), (8, 96), (32, 32), (64, 64), (97, 70), (128, 128), (160, 128),
                                   (200, 200)])
@pytest.mark.parametrize("amp", [1.0, 100.0])
def test_residual_against_64_bits_beside_outliers(nx, ny, amp):
    """The residual of the second sweep from P0 = noise of 1e-3 with a few nodes (some at the start of a
    block's rows, whatever the cluster's size) a thousand or more deviations away, against 64-bit sums
    over the pressures of the first two sweeps.  A warp's FP32 sums of squares are relative to its
    means of the sweep before, so their rounding (a square, its operand and eight additions, 2^-24
    each) is about 12 x 2^-24 of the whole variance, half of that in the root; P itself is rounded to 2^-24 on both sides
    and enters as a difference: 4 x 2^-24 more.  Together 6e-7; 2e-6 is allowed."""
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(nx)
    P0 = 1e-3 * rng.standard_normal((ny, nx))
    for C in (1, 2, 4, 8, 16):
        y = (C // 2) * -(-ny // C)
        P0[y if y < ny else 0, 0] = amp
    prob = uniform(nx, ny, bc=(1, 1, 1, 1), K=np.exp(rng.standard_normal((ny, nx))),
                   S0=0.2 + 0.5 * rng.random((ny, nx)), P0=P0)
    p = []
    for k in (0, 1):                          # the fields are those that the next sweep computes
        one = pkg.Solver.from_problem(prob, init_replay=k, fuse_sweeps=1)
        p.append(one.fields()[0].astype(np.float64))
        one.close()
    res = pkg.Solver.from_problem(prob, tol=0.0, max_sub_iters=2, check_every=2)
    assert res.fused_form() == pkg.FUSED_RESIDENT
    want = np.std(p[1] - p[0]) / np.std(p[1])
    assert res.init_stats.residual == pytest.approx(want, rel=2e-6)
    res.close()


@pytest.mark.parametrize("walls", ["periodic", "noflux"])
@pytest.mark.parametrize("every,cap", [(1, 20), (7, 70), (8, 68), (6, 100), (8, 4)])
def test_not_reported_where_a_solve_cannot_use_it(every, cap, walls):
    """A check period that is odd, or a cap that is no multiple of it: the host runs the solves, and the
    on-chip form is neither timed nor reported."""
    import paper_1808_07554_gb300 as pkg
    rng, prob = _problem(64, 64, walls)
    kw = dict(init_replay=0, tol=0.0, max_sub_iters=cap, check_every=every)
    one = pkg.Solver.from_problem(prob, fuse_sweeps=1, **kw)
    auto = pkg.Solver.from_problem(prob, **kw)
    assert auto.fused_form() != pkg.FUSED_RESIDENT
    assert all(r[0] != "resident" for r in auto.autotune_report())
    for s in (one, auto):
        st, stats = s.step(1)
        assert st == pkg.ENOTCONVERGED and stats[0].sub_iters == cap
    assert np.array_equal(one.get_state(), auto.get_state())
    one.close()
    auto.close()


def test_create_does_not_run_long_check_periods_to_time_the_form():
    """The form is timed over a bounded number of sweeps, so a handle with a check period of 4096 sweeps
    takes about as long to create as one with 64 (it took 17 times as long when it did not)."""
    import paper_1808_07554_gb300 as pkg
    rng, prob = _problem(64, 64, "noflux")
    took = {}
    for every in (64, 4096):
        for _ in range(4):
            t0 = time.perf_counter()
            s = pkg.Solver.from_problem(prob, init_replay=0, check_every=every, max_sub_iters=40960)
            took[every] = min(took.get(every, 1e9), time.perf_counter() - t0)
            assert any(r[0] == "resident" for r in s.autotune_report())
            s.close()
    assert took[4096] < 3 * took[64], took

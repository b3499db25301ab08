"""The kernels of a step outside the sub-iteration (S refresh, saturation update with the move of the
reference pressure, fields) compute wall nodes one per thread and the others four per thread.  On a
periodic lattice a problem rolled by some columns and rows is the same problem, with other nodes in the
edge and quad paths, so every plane of the state and every field must be the rolled one, bit for bit."""
import time

import numpy as np
import pytest

import workloads as W
from _problems import uniform

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_07554_gb300 import build
    build.build()
    import paper_1808_07554_gb300 as pkg
    pkg.load_library()


@pytest.mark.parametrize("lattice, D_c, warm", [(9, 0.0, 0), (9, 0.4, 1), (5, 0.4, 0)])
@pytest.mark.parametrize("nx, ny", [(8, 5), (9, 3), (9, 2), (12, 7), (13, 40), (132, 6), (133, 9),
                                    (520, 5), (646, 11)])
def test_rolled_problem_rolls_the_state(nx, ny, lattice, D_c, warm):
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(nx * 100 + ny)
    K, S0 = np.exp(0.5 * rng.standard_normal((ny, nx))), 0.2 + 0.5 * rng.random((ny, nx))
    Fp, Fs = rng.standard_normal((ny, nx)), 1e-2 * rng.standard_normal((ny, nx))
    Fp -= Fp.mean()

    def run(dy, dx):
        roll = lambda a: np.roll(a, (dy, dx), (0, 1))    # noqa: E731
        prob = uniform(nx, ny, K=roll(K), S0=roll(S0), Fp=roll(Fp), Fs=roll(Fs), mu_w=1.3, mu_n=5.0,
                       tau_mode=W.TAU_PHYSICAL_DT, dt=0.3 / nx ** 2)
        prob.sat_lattice, prob.D_c = lattice, D_c
        s = pkg.Solver.from_problem(prob, init_replay=16, warm_start=warm)
        for _ in range(2):
            s.step(1, replay=[16])
        out = [s.get_state(), *s.fields(), *s.velocity()]
        s.close()
        return out

    want = run(0, 0)
    for dy, dx in ((1, 1), (ny // 2, 2), (0, nx // 2 + 1)):
        for i, (a, b) in enumerate(zip(want, run(dy, dx))):
            assert np.array_equal(np.roll(a, (dy, dx), (-2, -1)), b), (i, dy, dx)


def test_timing_switched_between_steps():
    """set_timing before every step: the readings are there when it is on and only then, the states are
    those of an unswitched solver, and no graph is instantiated again (an instantiation takes as long as
    a step of this lattice: 112 us per step against 64 to 70)."""
    import paper_1808_07554_gb300 as pkg
    prob = W.quarter_five_spot(64, seed=2)
    make = lambda: pkg.Solver.from_problem(prob, init_replay=16, tol=0.0, max_sub_iters=16)   # noqa: E731
    plain, switched = make(), make()

    def median_step(s, mode):
        took = []
        for k in range(24):
            t0 = time.perf_counter()
            if mode == 2:
                s.set_timing(k % 2 == 0)
            st, stats = s.step(1)
            took.append(time.perf_counter() - t0)
            on = mode == 1 or (mode == 2 and k % 2 == 0)
            assert (stats[0].sweep_ms > 0 and stats[0].step_ms > 0) == on
        return float(np.median(took))

    best = {}
    for _ in range(4):
        for mode in (0, 1):
            plain.set_timing(mode == 1)
            best[mode] = min(best.get(mode, 1e9), median_step(plain, mode))
        for _ in range(2):
            best[2] = min(best.get(2, 1e9), median_step(switched, 2))
        assert np.array_equal(plain.get_state(), switched.get_state())
    assert best[2] < 1.3 * max(best[0], best[1]), best
    plain.close()
    switched.close()

"""The kernels of a step outside the sub-iteration (S refresh, saturation update with the move of the
reference pressure, fields) compute wall nodes one per thread and the others four per thread.  On a
periodic lattice a problem rolled by some columns and rows is the same problem, with other nodes in the
edge and quad paths, so every plane of the state and every field must be the rolled one, bit for bit."""
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

"""Four pressure sweeps per launch (one warp per tile of 56 columns) against one sweep per launch:
identical populations bit for bit, at the edges of its tiles: lattices narrower than a tile, one
column more or less than a whole number of tiles, odd widths (a wall in either column of a lane),
fewer rows than sweeps, wells on walls, at corners and at tile borders, dense sources, and walls
of both kinds on opposite sides."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("bc", [(1, 1, 1, 1), (2, 2, 2, 2), (1, 2, 2, 1), (2, 1, 1, 1)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (5, 1), (55, 9), (56, 8), (57, 7), (64, 64), (112, 5),
                                   (113, 131), (168, 33), (301, 257), (600, 40), (1237, 66)])
def test_four_sweeps_equal_single_sweeps(nx, ny, bc, dense):
    import paper_1808_07554_gb300 as pkg
    if ny < 3 and 2 in bc[2:]:
        pytest.skip("Dirichlet y-sides need three rows")
    rng = np.random.default_rng(nx * 1000 + ny)
    wells = {(0, 0), (nx - 1, ny - 1), (min(56, nx - 1), ny // 2), (min(55, nx - 1), ny // 3),
             (nx // 2, 0), (0, ny // 2)}
    prob = uniform(nx, ny, bc=bc, K=np.exp(rng.standard_normal((ny, nx))),
                   S0=0.2 + 0.5 * rng.random((ny, nx)),
                   Fp=rng.standard_normal((ny, nx)) if dense else None,
                   wells=[(i, j, 1e-2 * (1 + k), k % 2) for k, (i, j) in enumerate(sorted(wells))],
                   P_b=[rng.random(2 * (ny if s < 2 else nx) + 1) for s in range(4)],
                   S_b=[np.full(2 * (ny if s < 2 else nx) + 1, 0.3) for s in range(4)])
    one = pkg.Solver.from_problem(prob, init_replay=0, fuse_sweeps=1)
    four = pkg.Solver.from_problem(prob, init_replay=0, fuse_sweeps=4)
    assert four.fused_form() == pkg.FUSED_QUAD and four.sweep_config()[0] == 4
    state = one.get_state()
    state[:8] = 0.01 * rng.standard_normal(state[:8].shape)
    state[17] = 1.0 / (0.55 + 2.0 * rng.random(state[17].shape))
    state[19] = rng.standard_normal(state[19].shape)
    one.set_state(state)
    four.set_state(state)
    for n in (4, 9, 8):
        r1, r4 = one.pressure_sweeps(n), four.pressure_sweeps(n)
        assert np.array_equal(one.get_state(), four.get_state()), (n, nx, ny, bc)
        assert r4 == pytest.approx(r1, rel=1e-3, abs=1e-30)
    one.close()
    four.close()


@pytest.mark.parametrize("every, cap", [(8, 1024), (8, 1032), (8, 2056), (16, 3088), (1024, 3072)])
@pytest.mark.parametrize("fuse", [1, 4])
def test_graph_loop_equals_replay_across_moves_of_R(every, cap, fuse):
    """A solve of `cap` sweeps by the graph loop (the residual never meets the tolerance), with the
    reference pressure moved after 1024 and 2048 sweeps or, at 1024, never, against the same count
    driven from the host; then a second step, whose loop starts from the first one's conditions."""
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(cap)
    nx, ny = 70, 33
    prob = uniform(nx, ny, bc=(1, 1, 1, 1), K=np.exp(rng.standard_normal((ny, nx))), S0=0.4,
                   wells=[(0, 0, 1e-2, 0), (nx - 1, ny - 1, 1e-2, 1)])
    make = lambda: pkg.Solver.from_problem(prob, init_replay=16, check_every=every,   # noqa: E731
                                           max_sub_iters=cap, tol=0.0, fuse_sweeps=fuse)
    a, b = make(), make()
    for _ in range(2):
        st, stats = a.step(1)
        assert st == pkg.ENOTCONVERGED and stats[0].sub_iters == cap
        b.step(1, replay=[cap])
        assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


@pytest.mark.parametrize("bc", [(1, 1, 1, 1), (2, 2, 2, 2)])
@pytest.mark.parametrize("nx,ny,i,j", [(70, 33, 20, 10), (70, 33, 0, 0), (301, 257, 150, 128),
                                       (57, 9, 56, 4)])
def test_wells_that_share_a_node(nx, ny, i, j, bc):
    """Injectors and producers of one node: their sources are added up and then rounded once into the
    populations, with four sweeps per launch as with one, also in a batch."""
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(nx + i)
    prob = uniform(nx, ny, bc=bc, K=np.exp(rng.standard_normal((ny, nx))),
                   S0=0.2 + 0.5 * rng.random((ny, nx)),
                   wells=[(i, j, 0.1, 0), (i, j, 0.037, 1), (i, j, 0.0193, 0)],
                   P_b=[rng.random(2 * (ny if s < 2 else nx) + 1) for s in range(4)],
                   S_b=[np.full(2 * (ny if s < 2 else nx) + 1, 0.3) for s in range(4)])
    kw = dict(init_replay=0, tol=0.0, max_sub_iters=32)
    one = pkg.Solver.from_problem(prob, fuse_sweeps=1, **kw)
    four = pkg.Solver.from_problem(prob, fuse_sweeps=4, **kw)
    member = pkg.Solver.from_problem(prob, fuse_sweeps=4, **kw)
    with pkg.Batch([member]) as batch:
        for _ in range(2):
            one.step(1, replay=[32])
            four.step(1, replay=[32])
            batch.step(1, replay=[[32]])
            state = one.get_state()
            assert np.array_equal(state, four.get_state())
            assert np.array_equal(state, member.get_state())
    for s in (one, four, member):
        s.close()


@pytest.mark.parametrize("nx,ny", [(64, 64), (128, 128), (300, 140)])
def test_solves_driven_from_the_host_use_the_tuned_form(nx, ny):
    """A cap that is no multiple of check_every: the host runs the solve, four sweeps per launch where
    that is the form reported (lattices of fewer than 512^2 nodes included), and each check is a period of
    two launches and the reduction."""
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(nx)
    prob = uniform(nx, ny, bc=(1, 1, 1, 1), K=np.exp(rng.standard_normal((ny, nx))), S0=0.4,
                   wells=[(0, 0, 1e-2, 0), (nx - 1, ny - 1, 1e-2, 1)])
    kw = dict(init_replay=8, tol=0.0, check_every=8, max_sub_iters=44)
    one, auto = pkg.Solver.from_problem(prob, fuse_sweeps=1, **kw), pkg.Solver.from_problem(prob, **kw)
    if auto.fused_form() != pkg.FUSED_QUAD:
        pytest.skip("the four-sweep form was not the fastest here")
    before = auto.counters()
    assert one.step(1)[1][0].sub_iters == 44 and auto.step(1)[1][0].sub_iters == 44
    after = auto.counters()
    # refresh and saturation; five periods of 8 sweeps and one of 4, each with its reduction
    assert (after[0] - before[0], after[1] - before[1]) == (2 + 5 * 3 + 2, 44)
    assert np.array_equal(one.get_state(), auto.get_state())
    one.close()
    auto.close()


@pytest.mark.parametrize("bc", [(1, 1, 1, 1), (0, 0, 0, 0), (1, 1, 2, 1)])
@pytest.mark.parametrize("fuse", [0, 1, 2, 4])
def test_residual_of_a_last_sweep_on_its_own(fuse, bc):
    """A cap one sweep beyond a check, or a count one sweep beyond a move of R: the last sweep checks by
    itself and must compare with the increment of the sweep before it, over the same R.  Against the same
    count in one piece (equal states; the residual's sums are grouped differently: 1e-4), and, where R was
    moved, against a solve that does not move it (P is then rounded differently, by 1e-7 of it where it
    changes by 1e-4 and more per sweep: 1e-2)."""
    import paper_1808_07554_gb300 as pkg
    rng = np.random.default_rng(3)
    nx, ny = 70, 33
    prob = uniform(nx, ny, bc=bc, K=np.exp(rng.standard_normal((ny, nx))), S0=0.4,
                   wells=[(3, 2, 1e-2, 0), (nx - 4, ny - 3, 1e-2, 1)],
                   P_b=[rng.random(2 * (ny if s < 2 else nx) + 1) for s in range(4)],
                   S_b=[np.full(2 * (ny if s < 2 else nx) + 1, 0.3) for s in range(4)])
    make = lambda every, cap: pkg.Solver.from_problem(   # noqa: E731
        prob, init_replay=0, tol=0.0, check_every=every, max_sub_iters=cap, fuse_sweeps=fuse)
    for every, cap in ((8, 25), (7, 8), (2, 15), (16, 17), (1, 9)):
        a, b = make(every, cap), make(every, cap)
        (_, sa), (_, sb) = a.step(1), b.step(1, replay=[cap])
        assert sa[0].sub_iters == sb[0].sub_iters == cap
        assert np.array_equal(a.get_state(), b.get_state())
        assert sa[0].residual == pytest.approx(sb[0].residual, rel=1e-4), (every, cap)
        a.close()
        b.close()
    want = make(25, 1025)                     # R moves every 1025 sweeps: not within this solve
    r = want.step(1)[1][0].residual
    assert r > 1e-5
    for every, replay in ((8, None), (1, None), (8, [1025])):
        a = make(every, 1025)
        st = a.step(1, replay=replay)[1][0]
        assert st.sub_iters == 1025 and st.residual == pytest.approx(r, rel=1e-2), (every, replay)
        a.close()
    want.close()

"""Failure detection on the CUDA path, without faulting the GPU.

- Bounded grid-barrier waits: one block of the persistent solver kernel is made to leave
  at its first barrier without arriving (dg_test_barrier_fault), so the other blocks' wait
  runs out. The call must return DG_ERR_CUDA ("timed out") instead of hanging, and the
  device context must stay usable: after the hook is turned off the same mesh gives the
  result of a fresh one.
- Energy watchdog (dg_set_energy_watchdog): the kinetic energy of the scheme does not grow
  at nu = 0 under the CFL step (Sec. 2.2), so the watchdog stays quiet there; a step size far
  above the stability limit makes ||u||^2 grow and the call returns DG_ERR_UNSTABLE.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1808_04669_gb300 import build
    build.build()
    import paper_1808_04669_gb300 as pkg
    return pkg


def random_lattice(n_tri, k, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n_tri, (k + 1) * (k + 2) // 2, 2))


@pytest.mark.parametrize("precision,precond", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_barrier_timeout_is_reported_and_context_stays_usable(g, precision, precond):
    from paper_1808_04669_gb300 import DGError
    N, k = 32, 2
    vid, X = synth.split_square_mesh(N)
    v = random_lattice(2 * N * N, k, 5)
    mesh = g.DGMesh(vid, X, k, 1e-3, precision=precision, precond=precond)
    assert mesh.solver_stats()["blocks"] >= 2
    mesh.set_velocity(v)
    mesh.test_barrier_fault(spin_limit=1 << 14, skip_block=1)
    with pytest.raises(DGError) as e:
        mesh.project_divfree()
    assert e.value.code == -4 and "timed out" in str(e.value)
    # hook off: the same mesh works again and agrees with a fresh mesh
    mesh.test_barrier_fault(0, -1)
    mesh.set_velocity(v)
    mesh.project_divfree()
    mesh.rk3_step(0.01, 2)
    fresh = g.DGMesh(vid, X, k, 1e-3, precision=precision, precond=precond)
    fresh.set_velocity(v)
    fresh.project_divfree()
    fresh.rk3_step(0.01, 2)
    a, b = mesh.get_velocity(), fresh.get_velocity()
    assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()


def test_barrier_fault_hook_rejects_bad_arguments(g):
    from paper_1808_04669_gb300 import DGError
    vid, X = synth.split_square_mesh(2)
    mesh = g.DGMesh(vid, X, 1, 0.0)
    with pytest.raises(DGError):
        mesh.test_barrier_fault(-1, -1)
    with pytest.raises(DGError):
        mesh.test_barrier_fault(0, -2)


@pytest.mark.parametrize("precision", [0, 1])
def test_energy_watchdog_quiet_under_cfl_and_fires_above_it(g, precision):
    from paper_1808_04669_gb300 import DGError
    N, k = 16, 2
    vid, X = synth.split_square_mesh(N, L=1.0)
    v = random_lattice(2 * N * N, k, 11)
    dt = synth.cfl_dt(X, k, float(np.sqrt((v ** 2).sum(-1)).max()), 0.0)
    mesh = g.DGMesh(vid, X, k, 0.0, precision=precision)
    mesh.set_energy_watchdog(1e-10)
    mesh.set_velocity(v)
    mesh.project_divfree()
    E0 = mesh.diagnostics()["energy"]
    mesh.rk3_step(dt, 10)                    # stable: energy does not grow, no error
    assert mesh.diagnostics()["energy"] <= E0 * (1 + 1e-12)
    code = None
    for _ in range(30):                      # 40 x the CFL step: the unstable modes grow
        try:
            mesh.rk3_step(40 * dt, 1)
        except DGError as e:
            code = e.code
            assert "energy watchdog" in str(e)
            break
    assert code == -8
    # off again: the same oversized step no longer reports
    mesh.set_energy_watchdog(0.0)
    mesh.set_velocity(v)
    mesh.project_divfree()
    mesh.rk3_step(40 * dt, 1)


@pytest.mark.parametrize("precision,size0,dt0,size,dt", [(1, 1e8, 1e-2, 1.0, 1e-2), (1, 1e8, 1e-2, 1e-15, 1.0),
                                                         (1, 1e12, 1e-2, 1e9, 1e-13), (0, 1e8, 1e-2, 1.0, 1e-2),
                                                         (0, 1e70, 1e10, 1e-30, 1e20)])
def test_lattice_solve_drops_a_start_far_from_the_solution(g, precision, size0, dt0, size, dt):
    # a state that has nothing to do with the multipliers of the last steps, smaller by so much that
    # the residual of the extrapolated start overflows its sums or leaves its rounding in the result:
    # the steps agree with those of a fresh mesh. Both meet rtol 1e-13, so that they differ by that
    # times sqrt(cond(S)) (below 1e3 N), with a factor of ten to spare
    N, k = 16, 2
    vid, X = synth.split_square_mesh(N, L=1.0)
    mesh = g.DGMesh(vid, X, k, 0.0, precision=precision)
    fresh = g.DGMesh(vid, X, k, 0.0, precision=precision)
    mesh.set_velocity(size0 * random_lattice(2 * N * N, k, 5))
    mesh.step(dt0, 1, g.EULER)
    for m in (mesh, fresh):
        m.set_velocity(size * random_lattice(2 * N * N, k, 6))
    for _ in range(3):
        out = []
        for m in (mesh, fresh):
            m.step(dt, 1, g.EULER)
            out.append(m.get_velocity() / size)
        assert np.isfinite(out[1]).all()
        assert np.linalg.norm(out[0] - out[1]) < 1e-13 * np.sqrt(1e3 * N) * 10 * np.linalg.norm(out[1])


def check_good_state_after_overflow(mesh, fresh, v):
    # steps far above the stability limit, until a solve reports that its residual overflowed: nothing
    # of its multipliers stays, and a good state then gives the result of a fresh mesh
    from paper_1808_04669_gb300 import DGError
    mesh.set_velocity(v)
    mesh.project_divfree()
    code = 0
    for _ in range(10):
        try:
            mesh.rk3_step(10.0, 1)
        except DGError as e:
            code = e.code
            break
    assert code == -6
    for m in (mesh, fresh):
        m.set_velocity(v)
        m.rk3_step(1e-3, 2)
    a, b = mesh.get_velocity(), fresh.get_velocity()
    assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("precond", [1, 2])
def test_good_state_after_an_overflow(g, precond):
    N, k = 8, 2
    vid, X = synth.split_square_mesh(N, L=1.0, periodic=False)
    mesh, fresh = (g.DGMesh(vid, X, k, 0.0, precond=precond) for _ in range(2))
    check_good_state_after_overflow(mesh, fresh, random_lattice(2 * N * N, k, 1))


@pytest.mark.parametrize("precond", [0, 1])
def test_good_state_after_an_overflow_in_three_dimensions(g, precond):
    from synth.mesh3 import kuhn_cube_mesh
    vid, X = kuhn_cube_mesh(4)
    mesh, fresh = (g.DGMesh3(vid, X, 1, 0.0, precond=precond) for _ in range(2))
    check_good_state_after_overflow(mesh, fresh, np.random.default_rng(1).standard_normal((mesh.n_tet, mesh.n_lat, 3)))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("precond", [0, 1, 2])
def test_start_that_is_not_finite_is_dropped(g, precision, precond):
    # a step size 1e297 times the last one scales the start by as much: the residual's norm is inf - inf,
    # neither zero (mixed block Jacobi, whose refinement tests that norm alone, took it as converged) nor
    # the solve's failure. The step gives what it gives on a fresh mesh
    N, k = 8, 2
    vid, X = synth.split_square_mesh(N, L=1.0)
    v = random_lattice(2 * N * N, k, 1)
    mesh, fresh = (g.DGMesh(vid, X, k, 0.0, precision=precision, precond=precond) for _ in range(2))
    mesh.set_velocity(v)
    mesh.step(1e-300, 1, g.EULER)
    for m in (mesh, fresh):
        m.set_velocity(v)
        m.step(1e-3, 1, g.EULER)
    a, b = mesh.get_velocity(), fresh.get_velocity()
    assert np.linalg.norm(a - b) < 1e-13 * np.sqrt(1e3 * N) * 10 * np.linalg.norm(b)


def test_facet_solve_reports_a_right_hand_side_that_is_not_a_number(g):
    import torch
    from paper_1808_04669_gb300 import DGError
    vid, X = synth.split_square_mesh(4)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in g.host_facet_operator(vid, X, 1)]
    rhs = torch.zeros(t[0].shape[0], 2, dtype=torch.float64, device="cuda")
    rhs[3, 1] = float("nan")
    with pytest.raises(DGError) as e:
        g.facet_solve_noalloc(1, *t, rhs, torch.zeros_like(rhs))
    assert e.value.code == -6


@pytest.mark.parametrize("precision,precond", [(0, 1), (1, 1), (0, 2), (1, 2)])
@pytest.mark.parametrize("walls", [False, True])
def test_other_solvers_drop_a_start_far_from_the_solution(g, precision, precond, walls):
    # as above with the multilevel and block-Jacobi solvers: a state 1e8 times smaller than the last one,
    # then steps whose multipliers are again far smaller (the state is divergence-free by then)
    N, k = 16, 2
    vid, X = synth.split_square_mesh(N, L=1.0, periodic=not walls)
    mesh, fresh = (g.DGMesh(vid, X, k, 0.0, precision=precision, precond=precond) for _ in range(2))
    mesh.set_velocity(1e8 * random_lattice(2 * N * N, k, 5))
    mesh.step(1e-10, 1, g.EULER)
    for m in (mesh, fresh):
        m.set_velocity(random_lattice(2 * N * N, k, 6))
    for dt in (1e-10, 1e-4, 1e-4):
        out = []
        for m in (mesh, fresh):
            m.step(dt, 1, g.EULER)
            out.append(m.get_velocity())
        assert np.linalg.norm(out[0] - out[1]) < 1e-13 * np.sqrt(1e3 * N) * 10 * np.linalg.norm(out[1])


@pytest.mark.parametrize("precond", [0, 1])
def test_other_solvers_drop_a_start_far_from_the_solution_in_three_dimensions(g, precond):
    from synth.mesh3 import kuhn_cube_mesh
    N = 4
    vid, X = kuhn_cube_mesh(N)
    mesh, fresh = (g.DGMesh3(vid, X, 1, 0.0, precond=precond) for _ in range(2))
    rng = np.random.default_rng(1)
    mesh.set_velocity(1e8 * rng.standard_normal((mesh.n_tet, mesh.n_lat, 3)))
    mesh.rk3_step(1e-10, 1)
    v = rng.standard_normal((mesh.n_tet, mesh.n_lat, 3))
    for m in (mesh, fresh):
        m.set_velocity(v)
    for dt in (1e-10, 1e-4, 1e-4):
        out = []
        for m in (mesh, fresh):
            m.rk3_step(dt, 1)
            out.append(m.get_velocity())
        assert np.linalg.norm(out[0] - out[1]) < 1e-13 * np.sqrt(1e3 * N) * 10 * np.linalg.norm(out[1])

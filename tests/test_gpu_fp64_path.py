"""Both FP64 paths of FP64_EMULATED contexts against the oracle, each forced
(ehdg_set_fp64_path): the digit-split products on the tensor cores, which such a
context only runs by choice where a fixed-point form exists, and the kernels of
EHDG_FP64. Tolerance 1e-12 relative L2, the FP64 parity bound."""
import numpy as np
import pytest

from paper_1601_06681_gb300 import ehdg as E
from test_gpu_parity import OZAKI_CASES, RTOL, make_case, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")


def start(s, u0, g):
    if g is not None:
        s.set_boundary(g)
    s.set_state(u0)


@pytest.mark.parametrize("name", OZAKI_CASES)
@pytest.mark.parametrize("tensor_cores", [True, False])
def test_forced_path_matches_oracle(name, tensor_cores):
    mesh, p, kw, prob, u0, g = make_case(name)
    with E.Solver(mesh, p, tol=1e-10, max_iter=400, precision="fp64_emulated", **kw) as s:
        s.set_fp64_path(tensor_cores)
        start(s, u0, g)
        s.step_fixed(4)
        fixed, hist = s.get_state(), s.residual_history()
        start(s, u0, g)
        iters = s.run(2)
        u, uh = s.get_state()
    ou, ouh, ohist = prob.solve_step(u0, prob.trace(u0, g), g_new=g, fixed_iters=4)
    assert rel(fixed[0], ou) < RTOL and rel(fixed[1], ouh) < RTOL
    assert np.allclose(hist, ohist, rtol=1e-10, atol=1e-300)
    ou, ouh, oiters, _ = prob.run(u0, 2, g_of_t=None if g is None else (lambda t: g), tol=1e-10)
    assert iters == oiters
    assert rel(u, ou) < RTOL and rel(uh, ouh) < RTOL


@pytest.mark.parametrize("name", ["2d_be_const", "2d_cn_const", "3d_be_const_p3", "sw_be_p3"])
def test_path_changes_between_steps(name):
    """Steps on alternating paths, in one captured step graph after the other."""
    mesh, p, kw, prob, u0, g = make_case(name)
    with E.Solver(mesh, p, tol=1e-10, max_iter=400, precision="fp64_emulated", **kw) as s:
        start(s, u0, g)
        iters = []
        for k in range(4):
            s.set_fp64_path(k % 2 == 0)
            iters += s.run(1)
        u, uh = s.get_state()
    ou, ouh, oiters, _ = prob.run(u0, 4, g_of_t=None if g is None else (lambda t: g), tol=1e-10)
    assert iters == oiters
    assert rel(u, ou) < RTOL and rel(uh, ouh) < RTOL


@pytest.mark.parametrize("name", ["2d_be_const", "3d_be_const_p3_tiles", "sw_be_p3"])
@pytest.mark.parametrize("precision", ["tf32", "fp32"])
def test_tensor_core_outer_sweeps_reach_the_fp64_solution(name, precision):
    mesh, p, kw, prob, u0, g = make_case(name)
    with E.Solver(mesh, p, tol=1e-12, max_iter=400, precision=precision, inner_sweeps=6,
                  emulated_outer=True, **kw) as s:
        s.set_fp64_path(True)
        start(s, u0, g)
        s.run(2)
        u, uh = s.get_state()
    ou, ouh, _, _ = prob.run(u0, 2, g_of_t=None if g is None else (lambda t: g), tol=1e-13,
                             max_iter=2000)
    assert rel(u, ou) < 1e-10 and rel(uh, ouh) < 1e-10   # as the mixed forms are held elsewhere


def test_many_tiles_on_the_tensor_cores():
    """u = 1 + a.x - (a.beta) t is exact under backward Euler; 37,620 elements, the last
    tile ragged. Tolerance 1e-11: the stopping residual is 1e-13, the error at most 30
    times the last residual."""
    beta, a, dt = np.array([0.7, -0.4, 0.6]), np.array([0.3, -0.2, 0.5]), 5e-3
    sol = lambda x, t: 1.0 + x @ a - (a @ beta) * t      # noqa: E731
    with E.Solver(E.ehdg_mesh_structured((33, 34, 35)), 3, dt=dt, tol=1e-12, max_iter=500,
                  beta_const=beta, precision="fp64_emulated") as s:
        s.set_fp64_path(True)
        x, xf = s.node_coords(), s.face_point_coords()
        s.set_boundary(sol(xf, dt))
        s.set_state(sol(x, 0.0)[:, None, :])
        s.run(1)
        u, uh = s.get_state()
    assert np.abs(u[:, 0] - sol(x, dt)).max() < 1e-10
    assert np.abs(uh - sol(xf, dt)).max() < 1e-10


def test_contexts_without_the_path_are_refused():
    mesh, p, kw, prob, u0, g = make_case("2d_be_const")
    with E.Solver(mesh, p, **kw) as s:
        with pytest.raises(E.EhdgError) as ei:
            s.set_fp64_path(True)
        assert ei.value.status == 1

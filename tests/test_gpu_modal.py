"""The FP64 hexahedral step in Schur coefficients against the oracle: every
sign pattern of the velocity (each orients the axes' tables differently),
every degree, with forcing, backward Euler, Crank-Nicolson and steady, on
meshes of one element, of a single warp's ragged part and of several blocks.

Tolerance 1e-12 relative L2, the FP64 parity bound of the library: both sides
form the same iterates in float64, and a step's 30-odd contracting iterations
leave a few hundred roundings of 1.1e-16 at most."""
import numpy as np
import pytest

from paper_1601_06681_gb300 import ehdg as E
from paper_1601_06681_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("n,p,signs,scheme,force", [
    ((1, 1, 1), 3, (1, 1, 1), "be", False),
    ((2, 3, 2), 3, (-1, 1, 1), "cn", True),
    ((3, 2, 2), 3, (1, -1, -1), "be", True),
    ((2, 2, 3), 3, (-1, -1, -1), "steady", True),
    ((5, 4, 7), 2, (1, 1, -1), "be", False),
    ((3, 5, 2), 2, (-1, -1, 1), "cn", True),
    ((1, 33, 1), 2, (1, -1, 1), "steady", True),
    ((7, 6, 5), 1, (-1, 1, -1), "cn", True),
    ((1, 1, 65), 1, (1, 1, 1), "be", False),
])
def test_modal_step_matches_oracle(n, p, signs, scheme, force):
    from oracle import ehdg as O
    rng = np.random.default_rng(5)
    beta = np.array([0.9, 0.2, 0.5]) * np.array(signs)
    mesh = W.structured_mesh(n, lo=(0.0, -1.0, 0.5), hi=(1.0, 0.3, 2.5))
    dt, steps = 0.05, 2 if scheme != "steady" else 1
    prob = O.Problem(mesh, p, scheme=scheme, dt=dt, beta_const=beta)
    u0 = rng.standard_normal((prob.nel, 1, prob.Np))
    g = rng.standard_normal((prob.nface, prob.Nqf))
    f = rng.standard_normal(u0.shape) if force else None
    if scheme == "steady":
        u0 = np.zeros_like(u0)
    u_ref, uh_ref, iters, _ = O.Problem.run(prob, u0, steps, g_of_t=lambda t: g,
                                            f_of_t=(lambda t: f) if force else None, tol=1e-11)
    with E.Solver(mesh, p, scheme=scheme, dt=dt, tol=1e-11, beta_const=beta) as s:
        assert s.info["sum_factorised"] == 1
        s.set_boundary(g)
        if force:
            s.set_forcing(f)
        s.set_state(u0)
        got = s.run(steps)
        u, uh = s.get_state()
    assert got == iters
    assert rel(u, u_ref) < 1e-12
    assert rel(uh, uh_ref) < 1e-12


@pytest.mark.parametrize("n,p", [((55, 54, 53), 2), ((55, 54, 53), 3), ((33, 34, 35), 3)])
def test_linear_solution_is_exact_on_large_meshes(n, p):
    """u = 1 + a.x - (a.beta) t solves the equation and lies in the space, and
    backward Euler is exact for it, on meshes of over 4,864 tiles (one warp per
    tile, the last tile ragged) and below (a team per tile). Tolerance 1e-11: the
    step stops at a residual of 1e-13, the error is below 30 times the last
    residual for this iteration, and values are of order one."""
    beta, a, dt = np.array([0.7, -0.4, 0.6]), np.array([0.3, -0.2, 0.5]), 5e-3
    sol = lambda x, t: 1.0 + x @ a - (a @ beta) * t      # noqa: E731
    with E.Solver(E.ehdg_mesh_structured(n), p, dt=dt, tol=1e-13, max_iter=500,
                  beta_const=beta) as s:
        x, xf = s.node_coords(), s.face_point_coords()
        s.set_boundary(sol(xf, dt))
        s.set_state(sol(x, 0.0)[:, None, :])
        s.run(1)
        u, uh = s.get_state()
    assert np.abs(u[:, 0] - sol(x, dt)).max() < 1e-11
    assert np.abs(uh - sol(xf, dt)).max() < 1e-11


@pytest.mark.parametrize("p", [1, 2, 3])
def test_fixed_point_scales_exactly(p):
    """The sweep aligns each element to a power of two, so inputs scaled by a
    power of two (with the tolerance) give iterates scaled by it, far below and
    far above one. The step's and the reconstruction's FP64 sums scale exactly
    too, so equality is bit for bit."""
    n = (3, 4, 5)
    mesh = E.ehdg_mesh_structured(n)
    out = []
    for k in (0, -140, 90):
        with E.Solver(mesh, p, dt=1e-2, tol=np.ldexp(1e-11, k), beta_const=(0.7, -0.4, 0.6)) as s:
            rng = np.random.default_rng(3)
            s.set_boundary(np.ldexp(rng.standard_normal(s.trace_shape), k))
            s.set_state(np.ldexp(rng.standard_normal(s.state_shape), k))
            it = s.run(2)
            u, uh = s.get_state()
            out.append((it, np.ldexp(u, -k), np.ldexp(uh, -k)))
    for it, u, uh in out[1:]:
        assert it == out[0][0]
        assert np.array_equal(u, out[0][1]) and np.array_equal(uh, out[0][2])


@pytest.mark.parametrize("p", [1, 2, 3])
def test_zero_and_non_finite_states(p):
    """A zero state stays exactly zero; a state with a NaN ends as diverged and
    the context then still solves (a constant state stays constant)."""
    mesh = E.ehdg_mesh_structured((3, 3, 4))
    with E.Solver(mesh, p, dt=1e-2, tol=1e-11, beta_const=(0.7, -0.4, 0.6)) as s:
        s.set_boundary(np.zeros(s.trace_shape))
        s.set_state(np.zeros(s.state_shape))
        s.run(1)
        u, uh = s.get_state()
        assert not u.any() and not uh.any()
        bad = np.ones(s.state_shape)
        bad[5, 0, 0] = np.nan
        s.set_state(bad)
        with pytest.raises(E.EhdgError) as err:
            s.run(1)
        assert err.value.status == 5
        s.set_state(np.ones(s.state_shape))
        s.set_boundary(np.ones(s.trace_shape))
        s.run(1)
        u, uh = s.get_state()
        assert np.abs(u - 1).max() < 1e-12 and np.abs(uh - 1).max() < 1e-12


@pytest.mark.parametrize("n,p", [((55, 54, 53), 1), ((55, 54, 53), 2), ((33, 34, 35), 2),
                                 ((33, 34, 35), 3), ((3, 1, 11), 3)])
def test_crank_nicolson_keeps_a_linear_solution(n, p):
    """The same linear solution under Crank-Nicolson, which is exact for it too:
    the reconstruction 2 v - u^n in its three forms (one warp per tile, a team per
    tile, p = 1). Two steps; tolerance as above, twice for the factor 2."""
    beta, a, dt = np.array([0.7, -0.4, 0.6]), np.array([0.3, -0.2, 0.5]), 5e-3
    sol = lambda x, t: 1.0 + x @ a - (a @ beta) * t      # noqa: E731
    with E.Solver(E.ehdg_mesh_structured(n), p, scheme="cn", dt=dt, tol=1e-13, max_iter=500,
                  beta_const=beta) as s:
        x, xf = s.node_coords(), s.face_point_coords()
        s.set_boundary(sol(xf, 0.0))
        s.set_state(sol(x, 0.0)[:, None, :])
        for k in (1, 2):
            s.set_boundary(sol(xf, k * dt))
            s.run(1)
        u, uh = s.get_state()
    assert np.abs(u[:, 0] - sol(x, 2 * dt)).max() < 2e-11
    assert np.abs(uh - sol(xf, 2 * dt)).max() < 2e-11

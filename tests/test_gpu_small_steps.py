"""Elements fed from rest, where the operator's entries differ by orders of
magnitude: a small time step (a trace changes by dt |beta| / h of its inflow in a
sweep) and a velocity nearly along the faces that the data enters through. State
zero, two sweeps: the first ring of elements takes values of the small factor,
the second of its square, and each is compared with the oracle in terms of its
own size, face by face and element by element.

Tolerance 1e-12: the oracle's element solve is off by its condition number (a
mass matrix's, at most 1e3 up to p = 6) times 1.1e-16, in two sweeps; so is a
double evaluation of the same. Sums that keep 2^-56 of an operator's largest
entry, or of an element's largest value, are off by 1e-10 here.
Boundary data on outflow faces is zero, as the oracle's trace formula adds and
subtracts it."""
import numpy as np
import pytest

from paper_1601_06681_gb300 import ehdg as E
from paper_1601_06681_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")


def worst(a, b):
    """The largest relative L2 difference of a row (a face, an element) that is not zero in b."""
    a, b = a.reshape(len(b), -1), b.reshape(len(b), -1)
    n = np.linalg.norm(b, axis=1)
    assert np.all(np.abs(a[n == 0]) == 0)
    return (np.linalg.norm(a - b, axis=1)[n > 0] / n[n > 0]).max()


def two_sweeps(n, p, beta, dt, axis=None):
    """(uhat, u) of the library and of the oracle; axis: data on that axis's inflow faces only."""
    from oracle.ehdg import Problem
    beta = np.asarray(beta)
    mesh = W.structured_mesh(n)
    prob = Problem(mesh, p, scheme="be", dt=dt, beta_const=beta)
    fl = mesh["face_local"][:, 0]
    g = np.random.default_rng(1).uniform(0.5, 1.5, (prob.nface, prob.Nqf))
    g[beta[fl // 2] * (2 * (fl % 2) - 1) > 0] = 0.0
    if axis is not None:
        g[fl // 2 != axis] = 0.0
    u0 = np.zeros((prob.nel, 1, prob.Np))
    u_ref, uh_ref, _ = prob.solve_step(u0, prob.trace(u0, g), g_new=g, fixed_iters=2)
    with E.Solver(mesh, p, scheme="be", dt=dt, beta_const=beta) as s:
        s.set_boundary(g)
        s.set_state(u0)
        s.step_fixed(2)
        u, uh = s.get_state()
    return uh, u, uh_ref, u_ref


@pytest.mark.parametrize("p,beta,dt,axis", [
    (1, (0.8, 0.35), 1e-8, None),
    (2, (-0.8, 0.35), 1e-8, None),
    (4, (0.8, -0.35), 1e-8, None),
    (6, (-0.8, -0.35), 1e-8, None),
    (4, (0.8, 1e-7), 1e-2, 1),
    (3, (-1e-7, 0.6), 1e-2, 0),
])
def test_quadrilateral_traces_keep_their_own_digits(p, beta, dt, axis):
    uh, _, uh_ref, _ = two_sweeps((6, 5), p, beta, dt, axis)
    assert 0 < np.abs(uh_ref[uh_ref != 0]).min() < 1e-7
    assert worst(uh, uh_ref) < TOL


@pytest.mark.parametrize("p", [1, 2, 4])
def test_shallow_water_faces_do_not_take_the_other_velocity_s_unit(p):
    """Each element's fields are of sizes 1e-12 to 1 of their own; a face's trace holds phi
    and the normal velocity, and the other velocity, however large, only by dt squared."""
    from oracle.ehdg import Problem
    mesh = W.structured_mesh((6, 5), boundary_tag=W.TAG_WALL)
    prob = Problem(mesh, p, pde="sw", scheme="be", dt=1e-8, Phi=1.0)
    rng = np.random.default_rng(1)
    u0 = rng.standard_normal((prob.nel, 3, prob.Np)) * 10.0 ** rng.integers(-12, 1, (prob.nel, 3, 1))
    u_ref, uh_ref, _ = prob.solve_step(u0, prob.trace(u0), fixed_iters=2)
    with E.Solver(mesh, p, pde="sw", scheme="be", dt=1e-8, Phi=1.0) as s:
        s.set_state(u0)
        s.step_fixed(2)
        u, uh = s.get_state()
    assert worst(uh, uh_ref) < TOL
    assert worst(u, u_ref) < TOL


@pytest.mark.parametrize("p,beta,dt,axis", [
    (1, (0.8, 0.35), 1e-8, None),
    (6, (-0.8, -0.35), 1e-8, None),
    (4, (0.8, 1e-7), 1e-2, 1),
    (3, (-1e-7, 0.6), 1e-2, 0),
])
def test_quadrilateral_values_keep_their_own_digits(p, beta, dt, axis):
    _, u, _, u_ref = two_sweeps((6, 5), p, beta, dt, axis)
    assert worst(u, u_ref) < TOL


@pytest.mark.parametrize("p,beta,dt,axis", [
    (1, (0.8, 0.35, -0.5), 1e-8, None),
    (2, (-0.8, 0.35, 0.5), 1e-8, None),
    (3, (0.8, -0.35, 0.5), 1e-8, None),
    (2, (0.8, 1e-7, -0.6), 1e-2, 1),
    (3, (-0.8, 0.6, 1e-7), 1e-2, 2),
])
def test_hexahedral_traces_and_values_keep_their_own_digits(p, beta, dt, axis):
    uh, u, uh_ref, u_ref = two_sweeps((3, 4, 2), p, beta, dt, axis)
    assert worst(uh, uh_ref) < TOL
    assert worst(u, u_ref) < TOL


@pytest.mark.parametrize("p", [1, 3, 5])
@pytest.mark.parametrize("k", [0, 23])
def test_shallow_water_fields_of_different_size(p, k):
    """With Phi = 4^k the wave speed is 2^k and phi is 2^k times the velocities: the
    problem with Phi = 1 in other units, so its fields and traces are the oracle's
    there times powers of two. 2^23 is far beyond a geopotential of 1e5 m^2/s^2, and
    a sum that holds the velocities in units of phi's last place shows there.
    Tolerance 1e-12, the FP64 parity bound, per field."""
    from oracle.ehdg import Problem
    mesh = W.structured_mesh((6, 5), boundary_tag=W.TAG_WALL)
    dt, c = 2.0 ** -9, 2.0 ** k
    prob = Problem(mesh, p, pde="sw", scheme="be", dt=dt, Phi=1.0)
    u0 = np.random.default_rng(2).standard_normal((prob.nel, 3, prob.Np))
    u_ref, uh_ref, _ = prob.solve_step(u0, prob.trace(u0), fixed_iters=3)
    scale = np.array([c, 1.0, 1.0])[None, :, None]
    with E.Solver(mesh, p, pde="sw", scheme="be", dt=dt / c, Phi=c * c) as s:
        s.set_state(u0 * scale)
        s.step_fixed(3)
        u, uh = s.get_state()
    u, uh = u / scale, uh / c
    assert np.linalg.norm(uh - uh_ref) < TOL * np.linalg.norm(uh_ref)
    for f in range(3):
        assert np.linalg.norm(u[:, f] - u_ref[:, f]) < TOL * np.linalg.norm(u_ref[:, f])

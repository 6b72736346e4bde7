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

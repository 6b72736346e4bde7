"""The tile-shape choice (ehdg_autotune_sweep_tile) where the sum-factorised FP64
sweep still runs, and where the sweep in Schur coefficients has taken its place."""
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


@pytest.mark.parametrize("n,p,beta,precision", [
    ((6, 5, 4), 1, (0.7, -0.5, 0.4), "fp32"),
    ((6, 5, 4), 2, (0.7, 0.5, 0.4), "tf32"),
    ((5, 3, 4), 3, (0.3, -1.0, 0.6), "bf16"),
    ((7, 5, 4), 2, (0.7, 0.0, 0.0), "fp64"),
])
def test_tile_choice_of_the_sum_factorised_sweep_keeps_iterates(n, p, beta, precision):
    """Mixed precision on hexahedra and a velocity along the faces run the FP64 sweep
    whose tile is chosen; a row is one thread's chain for any tile, so the iterates of
    the outer sweeps and of the corrections between them are equal bit for bit."""
    mesh = W.structured_mesh(n)
    rng = np.random.default_rng(4)
    states = []
    with E.Solver(mesh, p, dt=0.02, tol=1e-11, max_iter=300, beta_const=beta, precision=precision,
                  inner_sweeps=0 if precision == "fp64" else 4) as s:
        assert s.info["sum_factorised"] == 1
        g, u0 = rng.standard_normal(s.trace_shape), rng.standard_normal(s.state_shape)
        for ft in (2, 4, 8):
            best, ms = s.autotune_sweep_tile((ft,))
            assert best == ft and ms > 0
            s.set_boundary(g)
            s.set_state(u0)
            s.step_fixed(5)
            states.append(s.get_state())
    for a in states[1:]:
        assert np.array_equal(a[0], states[0][0]) and np.array_equal(a[1], states[0][1])


def test_choice_stays_where_the_sweep_has_no_tile():
    """FP64 on hexahedra: the candidates are the same step, so no timing decides."""
    with E.Solver(W.structured_mesh((4, 3, 3)), 2, dt=0.02, beta_const=(0.7, -0.5, 0.4)) as s:
        s.set_boundary(np.ones(s.trace_shape))
        s.set_state(np.ones(s.state_shape))
        for ft in (8, 2, 4, 8):
            assert s.autotune_sweep_tile((3, ft))[0] == ft
            for _ in range(3):
                best, ms = s.autotune_sweep_tile()
                assert best == ft and ms > 0

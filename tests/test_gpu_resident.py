"""The forms of a step's iterations on quadrilaterals with one shared operator:
one cluster of blocks (up to 16 tiles of 128 elements), one resident block per
tile, several tiles per block. Each forms the same integers and the same sums as
the launch per iteration, so a converged step equals the same number of single
sweeps bit for bit, residuals included."""
import numpy as np
import pytest

from paper_1601_06681_gb300 import ehdg as E

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")


@pytest.mark.parametrize("n,p,signs", [
    ((1, 1), 1, (1, 1)),
    ((16, 8), 2, (-1, 1)),        # one whole tile
    ((43, 3), 3, (1, -1)),        # one element in the second tile
    ((64, 32), 6, (-1, -1)),      # 16 tiles: the largest cluster
    ((683, 3), 4, (1, 1)),        # one element more
    ((260, 240), 4, (-1, 1)),     # more tiles than resident blocks
])
@pytest.mark.parametrize("scheme", ["be", "cn"])
def test_converged_step_equals_single_sweeps(n, p, signs, scheme):
    rng = np.random.default_rng(7)
    beta = np.array([0.8, 0.35]) * np.array(signs)
    with E.Solver(E.ehdg_mesh_structured(n), p, scheme=scheme, dt=5e-3, tol=1e-10, max_iter=500,
                  beta_const=beta) as s:
        g, u0 = rng.standard_normal(s.trace_shape), rng.standard_normal(s.state_shape)
        out = []
        for fixed in (0, 1):
            s.set_boundary(g)
            s.set_state(u0)
            if fixed:
                s.step_fixed(out[0][0])
                it = out[0][0]
            else:
                it = s.run(1)[0]
            out.append((it, s.residual_history()[:it].copy(), *s.get_state()))
    assert out[0][0] > 1
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)


def test_not_converged_and_non_finite_in_a_cluster():
    mesh = E.ehdg_mesh_structured((20, 20))
    with E.Solver(mesh, 2, dt=1e-2, tol=1e-12, max_iter=3, beta_const=(0.7, -0.4)) as s:
        s.set_boundary(np.ones(s.trace_shape))
        u0 = np.random.default_rng(1).standard_normal(s.state_shape)
        s.set_state(u0)
        with pytest.raises(E.EhdgError):
            s.run(1)
        assert s.residual_history().size == 3
        u0[7, 0, 0] = np.inf
        s.set_state(u0)
        with pytest.raises(E.EhdgError) as err:
            s.run(1)
        assert err.value.status == 5

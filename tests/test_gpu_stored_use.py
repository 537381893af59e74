"""Which solves run the coarse cycle as a stored matrix, as their statistics tell it."""
import numpy as np
import pytest

from fem_inputs import problems as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def B():
    from paper_1503_01287_gb300 import binding
    return binding


def handle(prob, **o):
    return B().setup_problem(prob, B().default_options(**o))


def solve(h, prob, tol=1e-8):
    b = torch.from_numpy(np.ascontiguousarray(prob.rhs())).cuda()
    x = torch.zeros_like(b)
    st = h.solve(b, x, tol, True)
    assert st.converged
    return st


@pytest.mark.parametrize("make,opts,stored", [
    (lambda: fp.vector_laplace_problem(1, seed=0), {}, 0),               # a single level
    (lambda: fp.vector_laplace_problem(3, seed=0), {}, 1),
    (lambda: fp.elasticity_problem((4, 5, 3), seed=1), {"precision": 1}, 1),
    (lambda: fp.elasticity_problem(9, seed=3, nu=0.4), {}, 2),
    (lambda: fp.elasticity_problem(9, seed=3, nu=0.4), {"precision": 2}, 2),
    (lambda: fp.elasticity_problem(9, seed=3, nu=0.4), {"cluster_from": 0}, 0),
    (lambda: fp.elasticity_problem(9, seed=3, nu=0.4), {"gs_cluster": 0}, 0),
    (lambda: fp.elasticity_problem(9, seed=3, nu=0.499), {}, 0),          # block condition
    (lambda: fp.mixed_elasticity_problem(6, nu=0.49, seed=4), {}, 2),
    (lambda: fp.mixed_elasticity_problem(6, nu=0.49, seed=4), {"smoother": 4}, 0),
    (lambda: fp.stokes_lid_problem(7), {"precision": 1}, 0)])
def test_statistics_name_the_stored_level(make, opts, stored):
    prob = make()
    h = handle(prob, max_iterations=1, **opts)
    b = torch.from_numpy(np.ascontiguousarray(prob.rhs())).cuda()
    st = h.solve(b, torch.zeros_like(b), 1e-8, True)
    assert st.stored_from == stored


@pytest.mark.parametrize("precision,tile,size,stored", [
    (1, -1, (4, 5, 3), 1), (1, -1, 9, 2), (1, 0, 9, 0), (0, -1, 9, 0)])
def test_batched_statistics_name_the_stored_level(precision, tile, size, stored):
    prob = fp.elasticity_problem(size, seed=3)
    h = handle(prob, precision=precision, batch_tile=tile)
    b = torch.from_numpy(np.ascontiguousarray(prob.rhs())).cuda()
    x = torch.zeros_like(b)
    rc, st = B().solve_batched([h], [b], [x], 1, 1e-8)
    assert rc == 0 and st[0].stored_from == stored

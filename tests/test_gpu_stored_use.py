"""Which solves run the coarse cycle as a stored matrix, as their statistics tell it."""
import os

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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("size", [3, 9, 11])       # stored: level 0, level 1, more than 4,096
def test_weight_changes(size, precision):
    """Under new weights the cycle runs operation by operation, and repeated solves bring the
    same stored level back; under the weights that the matrix holds it is in use at once."""
    prob = fp.elasticity_problem(size, seed=3)
    h, ops = handle(prob, precision=precision), handle(prob, precision=precision,
                                                       cluster_from=0, cycle_kernel=1)
    level = solve(h, prob).stored_from
    assert level == (1 if size == 3 else 2)
    h.set_weights(0.9, 1.1, 1.0)
    ops.set_weights(0.9, 1.1, 1.0)
    assert solve(h, prob).stored_from == 0
    h.set_weights(1.0, 1.0, 1.0)
    assert solve(h, prob).stored_from == level
    h.set_weights(0.9, 1.1, 1.0)
    want = solve(ops, prob).iterations
    seen = []
    for _ in range(10):
        st = solve(h, prob)
        assert abs(st.iterations - want) <= 1
        seen.append(st.stored_from)
    assert seen[0] == 0 and seen[-1] == level and seen == sorted(seen)
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(prob.n_dof)).cuda()
    r[torch.from_numpy(np.repeat((prob.tags & fp.TAG_DIRICHLET) != 0, 3)).cuda()] = 0.0
    z, ref = torch.zeros_like(r), torch.zeros_like(r)
    h.apply_preconditioner(r, z)
    ops.apply_preconditioner(r, ref)
    # as in the tests of the stored cycle: at most 1000 (FP32: 200) roundings
    tol = 1000 * 2.0 ** -53 if precision == 0 else 200 * 2.0 ** -24
    assert float((z - ref).norm() / ref.norm()) <= tol


@pytest.mark.parametrize("size,precision", [((4, 5, 3), 0), ((4, 5, 3), 1), (11, 0), (11, 1)])
def test_a_weight_change_is_a_copy(size, precision):
    """No matrix is filled by a change of weights itself (2 to 20 ms): well below 1 ms."""
    import time
    h = handle(fp.elasticity_problem(size, seed=3), precision=precision)
    best = 1.0
    for k in range(20):
        t = time.perf_counter()
        h.set_weights(0.9 + 0.01 * k, 1.1, 1.0)
        best = min(best, time.perf_counter() - t)
    assert best < 1e-3


@pytest.mark.parametrize("size", [9, 12])          # 12: the batch has a matrix of its own
def test_batched_weight_changes(size):
    prob = fp.elasticity_problem(size, seed=3)
    h = handle(prob, precision=1)
    b = torch.from_numpy(np.ascontiguousarray(prob.rhs())).cuda()
    x = torch.zeros_like(b)

    def stored():
        rc, st = B().solve_batched([h], [b], [x], 1, 1e-8)
        assert rc == 0
        return st[0].stored_from

    level = stored()
    assert level > 0
    h.set_weights(0.9, 1.1, 1.0)
    seen = [stored() for _ in range(6)]
    assert seen[0] == 0 and seen[-1] == level
    h.set_weights(1.0, 1.0, 1.0)
    assert stored() == 0
    h.set_weights(0.9, 1.1, 1.0)
    assert stored() == level


@pytest.mark.parametrize("size", [3, 11])
def test_weights_set_after_setup(size):
    """The matrix is filled for the weights that a program sets before its first solve, and
    once only."""
    prob = fp.elasticity_problem(size, seed=3)
    h = handle(prob, precision=1)
    h.set_weights(0.9, 1.1, 1.0)
    assert solve(h, prob).stored_from > 0
    h = handle(prob, precision=1)
    h.set_weights(0.9, 1.1, 1.0)
    h.set_weights(0.8, 1.1, 1.0)
    assert solve(h, prob).stored_from == 0
    h.set_weights(0.9, 1.1, 1.0)
    assert solve(h, prob).stored_from > 0


def test_learned_weights_are_stored():
    prob = fp.elasticity_problem((4, 5, 3), seed=1)
    h = handle(prob, precision=1)
    solve(h, prob)
    theta = np.load(os.path.join(os.path.dirname(B().__file__), "weights", "mlp_theta.npy"))
    h.learn_weights(theta)
    assert solve(h, prob).stored_from == 1


def test_a_failing_probe_leaves_the_weights():
    """learn_weights on a saddle handle whose Krylov method its probe solves refuse."""
    prob = fp.mixed_elasticity_problem(4, nu=0.45, seed=4)
    h = handle(prob, krylov=B().AMG_KRYLOV_PCG)
    h.set_weights(0.8, 1.2, 0.7)
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(prob.n_dof)).cuda()
    z, again = torch.zeros_like(r), torch.zeros_like(r)
    h.apply_preconditioner(r, z)
    w = h.weights()
    with pytest.raises(Exception):
        h.learn_weights(np.zeros(B().MLP_NPARAM, dtype=np.float32))
    assert np.array_equal(h.weights(), w)
    h.apply_preconditioner(r, again)
    assert torch.equal(z, again)

"""The cycle below a level as one stored matrix (default options) against the same cycle
run operation by operation (cluster_from = 0, cycle_kernel = 1): one preconditioner
application and a solve, at the sizes where the stored level or its tiles change."""
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


PROBLEMS = {
    "laplace_1": lambda: fp.vector_laplace_problem(1, seed=0),          # a single level
    "laplace_3": lambda: fp.vector_laplace_problem(3, seed=0),          # level 0 stored
    "elasticity_4x5x3": lambda: fp.elasticity_problem((4, 5, 3), seed=1),
    "elasticity_7x6x7": lambda: fp.elasticity_problem((7, 6, 7), seed=2),
    "elasticity_9": lambda: fp.elasticity_problem(9, seed=3, nu=0.4),   # level 1 stored
    "mixed_4": lambda: fp.mixed_elasticity_problem(4, nu=0.45, seed=4),
    "mixed_6": lambda: fp.mixed_elasticity_problem(6, nu=0.49, seed=4),
    "stokes_5": lambda: fp.stokes_lid_problem(5),
}

# One application chains at most a few hundred roundings of size 2^-53 or 2^-24 (the
# colours of every level, down and up); their sum stays below 1000 units of the result.
TOL = {0: 1000 * 2.0 ** -53, 1: 200 * 2.0 ** -24, 2: 200 * 2.0 ** -24}


def residual_like(prob, seed):
    r = np.random.default_rng(seed).standard_normal(prob.n_dof)
    r[:3 * prob.n_nodes][np.repeat((prob.tags & fp.TAG_DIRICHLET) != 0, 3)] = 0.0
    return torch.from_numpy(r).cuda()


def pair(prob, **o):
    return (B().setup_problem(prob, B().default_options(**o)),
            B().setup_problem(prob, B().default_options(cluster_from=0, cycle_kernel=1, **o)))


def apply(h, r):
    z = torch.zeros_like(r)
    h.apply_preconditioner(r, z)
    return z


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name,opts", [
    ("laplace_1", {}), ("laplace_3", {}), ("elasticity_4x5x3", {}), ("elasticity_7x6x7", {}),
    ("elasticity_9", {}), ("elasticity_9", {"nu": 2}), ("elasticity_4x5x3", {"cycles": 2}),
    ("elasticity_9", {"smoother": 1, "m_pre": 2}), ("elasticity_9", {"m_pre": 0, "m_post": 2}),
    ("elasticity_9", {"post_order": 1}),
    ("mixed_4", {}), ("mixed_6", {"nu": 2}), ("mixed_6", {"smoother": 3}), ("stokes_5", {}),
    ("stokes_5", {"smoother": 3, "cycles": 2})])
def test_stored_cycle_matches_operations(name, opts, precision):
    prob = PROBLEMS[name]()
    h, ops = pair(prob, precision=precision, **opts)
    r = residual_like(prob, 5)
    z, ref = apply(h, r), apply(ops, r)
    assert float((z - ref).norm() / ref.norm()) <= TOL[precision]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", ["laplace_3", "elasticity_9", "mixed_6"])
def test_weights_reach_the_stored_cycle(name, precision):
    """New weights on every level change the stored matrix, also for graphs captured before;
    setting the first weights again restores the first results."""
    prob = PROBLEMS[name]()
    h, ops = pair(prob, precision=precision)
    r = residual_like(prob, 6)
    b = torch.from_numpy(prob.rhs()).cuda()
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    first = apply(h, r)
    h.solve(b, x, 1e-8, True)
    for q in (h, ops):
        q.set_weights(0.8, 1.2, 0.7)
    z, ref = apply(h, r), apply(ops, r)
    assert float((z - ref).norm() / ref.norm()) <= TOL[precision]
    assert float((z - first).norm() / ref.norm()) > 1e-3
    sa, sb = h.solve(b, x, 1e-8, True), ops.solve(b, y, 1e-8, True)
    assert sa.converged and abs(sa.iterations - sb.iterations) <= 1
    h.set_weights(1.0, 1.0, 1.0)
    assert torch.equal(apply(h, r), first)


@pytest.mark.parametrize("precision", [0, 1])
def test_weights_replace_a_large_stored_cycle(precision):
    """A stored level of more than 4,096 unknowns (11^3: 5,202 on level 1) gives way to a
    smaller one when its weights change, also for the captured CG loop."""
    prob = fp.elasticity_problem(11, seed=3)
    h, ops = pair(prob, precision=precision)
    assert 4096 < 3 * h.level_info(1).n_nodes <= 6144
    r = residual_like(prob, 6)
    b = torch.from_numpy(prob.rhs()).cuda()
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    for w in ((1.0, 1.0, 1.0), (0.9, 1.1, 1.0), (1.0, 1.0, 1.0)):
        for q in (h, ops):
            q.set_weights(*w)
        z, ref = apply(h, r), apply(ops, r)
        assert float((z - ref).norm() / ref.norm()) <= TOL[precision]
        sa, sb = h.solve(b, x, 1e-8, True), ops.solve(b, y, 1e-8, True)
        assert sa.converged and abs(sa.iterations - sb.iterations) <= 1


def test_linear_and_repeatable():
    """M (a u + v) = a M u + M v within rounding, and equal bits on repetition."""
    prob = PROBLEMS["elasticity_9"]()
    h = B().setup_problem(prob, B().default_options(precision=0))
    u, v = residual_like(prob, 7), residual_like(prob, 8)
    zu, zv, zs = apply(h, u), apply(h, v), apply(h, 3.0 * u + v)
    assert float((zs - 3.0 * zu - zv).norm() / zs.norm()) <= TOL[0]
    assert torch.equal(apply(h, u), zu)


@pytest.mark.parametrize("n_rhs", [1, 16])
@pytest.mark.parametrize("size", [3, (4, 5, 3), 8, (10, 11, 9), 12])
def test_batched_stored_cycle(size, n_rhs):
    """Batched FP32 solves through the stored cycle (level 0, level 1, and a batch-only one
    below the single solve's) against batched solves without it (batch_tile given): the same
    iteration counts within one and the same solutions to the solver's tolerance."""
    prob = fp.elasticity_problem(size, seed=9, nu=0.35)
    rng = np.random.default_rng(10)
    b = rng.standard_normal((n_rhs, 3 * prob.n_nodes))
    b[:, np.repeat((prob.tags & fp.TAG_DIRICHLET) != 0, 3)] = 0.0
    b = torch.from_numpy(b).cuda()
    out = []
    for tile in (-1, 0):
        h = B().setup_problem(prob, B().default_options(precision=1, batch_tile=tile))
        for w in ((1.0, 1.0, 1.0), (0.9, 1.1, 1.0)):    # the batch's own matrix follows too
            h.set_weights(*w)
            x = torch.zeros_like(b)
            rc, st = B().solve_batched([h], [b], [x], n_rhs, 1e-9)
            assert rc == 0
            out.append((x, st[0].iterations))
    for k in (0, 1):
        assert abs(out[k][1] - out[2 + k][1]) <= 1
        assert float((out[k][0] - out[2 + k][0]).norm() / out[2 + k][0].norm()) <= 1e-7

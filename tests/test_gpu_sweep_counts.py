"""Cycles with 0, 1 and 2 pre- and post-smoothing sweeps, one and two cycles, V and W, against
the oracle: the sweeps from x = 0 that read half of A, the residual seeded by them, and the
segregated Gauss-Seidel sweeps that alternate between two vectors; CG on systems smaller than
one thread block."""
import numpy as np
import pytest

from fem_inputs import problems as fp
from oracle import amg

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


PROBLEMS = {"elasticity": (lambda: fp.elasticity_problem((5, 4, 6), seed=7), "gs", 0),
            "jacobi": (lambda: fp.elasticity_problem((5, 4, 6), seed=7), "jacobi", 1),
            "mixed": (lambda: fp.mixed_elasticity_problem(4, nu=0.47, seed=5), "sgs", 2),
            "braess": (lambda: fp.mixed_elasticity_problem(4, nu=0.47, seed=5), "bs", 3)}


@pytest.mark.parametrize("cluster_from,cycle_kernel", [(-1, 0), (0, 1), (0, 2)])
@pytest.mark.parametrize("m_pre,m_post,nu,cycles", [
    (1, 1, 1, 1), (0, 1, 1, 1), (0, 2, 1, 1), (2, 0, 1, 1), (1, 2, 2, 1), (2, 1, 2, 1),
    (1, 1, 1, 2), (2, 2, 2, 2)])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_sweep_counts(name, m_pre, m_post, nu, cycles, cluster_from, cycle_kernel):
    make, smoother, code = PROBLEMS[name]
    prob = make()
    kw = dict(m_pre=m_pre, m_post=m_post, nu=nu, cycles=cycles)
    h = B().setup_problem(prob, B().default_options(smoother=code, cluster_from=cluster_from,
                                                    cycle_kernel=cycle_kernel, **kw))
    oh = amg.build_hierarchy(prob, amg.Options(smoother=smoother, **kw))
    w = np.ones((h.n_levels, 3))
    w[0] = (0.9, 1.1, 0.8)          # weights other than 1: the seed (1 - omega) s is not zero
    h.set_level_weights(w)
    oh.opts.level_weights = [tuple(q) for q in w]
    r = np.random.default_rng(3).standard_normal(prob.n_dof)
    z = torch.zeros(prob.n_dof, dtype=torch.float64, device="cuda")
    h.apply_preconditioner(torch.from_numpy(r).cuda(), z)
    want = amg.precondition(oh, r)
    # the parity tests' bound for one FP64 preconditioner application
    assert np.all(np.abs(z.cpu().numpy() - want) <= 1e-10 * np.abs(want).max())


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 2, (1, 3, 2), 5])
def test_small_cg(n, precision):
    """The CG reductions with fewer nodes than a block (27) up to a few blocks."""
    prob = fp.elasticity_problem(n, seed=4)
    h = B().setup_problem(prob, B().default_options(precision=precision))
    b = torch.from_numpy(prob.rhs()).cuda()
    x = torch.zeros_like(b)
    for _ in range(2):                     # the captured loop, then its replay
        st = h.solve(b, x, 1e-10, True)
        assert st.converged
        ref, _ = amg.solve(prob, tol=1e-13)
        assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-8 * np.linalg.norm(ref.x)

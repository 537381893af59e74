"""The stored coarse cycle rounds like the operations that it stands for: its FP32 error
against the FP64 cycle over several residuals, and in FP64 the difference between the two."""
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
    "laplace_3": (lambda: fp.vector_laplace_problem(3, seed=0), {}),
    "elasticity_4x5x3": (lambda: fp.elasticity_problem((4, 5, 3), seed=1), {}),
    "elasticity_9": (lambda: fp.elasticity_problem(9, seed=3), {}),
    "elasticity_9_nu49": (lambda: fp.elasticity_problem(9, seed=3, nu=0.49), {}),
    "elasticity_11": (lambda: fp.elasticity_problem(11, seed=3), {}),   # 5,202 unknowns stored
    "mixed_6": (lambda: fp.mixed_elasticity_problem(6, nu=0.49, seed=4), {}),
    "mixed_6_bs": (lambda: fp.mixed_elasticity_problem(6, nu=0.49, seed=4), {"smoother": 3}),
}
OPS = {"cluster_from": 0, "cycle_kernel": 1}


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_rounds_like_the_operations(name):
    make, opts = PROBLEMS[name]
    prob = make()
    rng = np.random.default_rng(12)
    fixed = np.repeat((prob.tags & fp.TAG_DIRICHLET) != 0, 3)
    residuals = []
    for _ in range(12):
        r = rng.standard_normal(prob.n_dof)
        r[:3 * prob.n_nodes][fixed] = 0.0
        residuals.append(torch.from_numpy(r).cuda())

    def apply(**o):
        h = B().setup_problem(prob, B().default_options(**opts, **o))
        out = []
        for r in residuals:
            z = torch.zeros_like(r)
            h.apply_preconditioner(r, z)
            out.append(z)
        return out

    def rms(got, want):
        return np.sqrt(np.mean([float((a - b).norm() / b.norm()) ** 2
                                for a, b in zip(got, want)]))

    ref = apply(precision=0, **OPS)
    # two FP64 roundings of a cycle of a few hundred operations: tens of units 2^-53 at most
    # (an FP64 sum of the blocks in another order alone moves it by 1 to 5)
    assert rms(apply(precision=0), ref) <= 40 * 2.0 ** -53
    # a matrix built in plain FP32 doubles the error (7.1e-7 against 3.4e-7 at 32^3)
    assert rms(apply(precision=1), ref) <= 1.5 * rms(apply(precision=1, **OPS), ref)

"""The FP32 preconditioner of Stokes systems, whose K is singular: its error against the FP64
cycle, constant pressure taken out, is that of the cycle run operation by operation."""
import numpy as np
import pytest

from fem_inputs import problems as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def B():
    from paper_1503_01287_gb300 import binding
    return binding


def handle(prob, **o):
    h = B().setup_problem(prob, B().default_options(**o))
    h.set_pressure_weights(np.ascontiguousarray(prob.p_weights))
    return h


# two roundings of one cycle: their errors over 16 residuals are alike within a factor 2
@pytest.mark.parametrize("smoother", [2, 3])
@pytest.mark.parametrize("n", [5, 6, 7])
def test_fp32_error_is_that_of_the_operations(n, smoother):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    prob = fp.stokes_lid_problem(n)
    nu = 3 * prob.n_nodes
    w = torch.from_numpy(np.ascontiguousarray(prob.p_weights)).cuda()
    free = torch.from_numpy(np.repeat((prob.tags & fp.TAG_DIRICHLET) == 0, 3)).cuda()
    ref = handle(prob, smoother=smoother, cluster_from=0, cycle_kernel=1)
    rng = np.random.default_rng(8)
    residuals = []
    for _ in range(16):
        x = torch.from_numpy(rng.standard_normal(prob.n_dof)).cuda()
        x[:nu] *= free
        y = torch.zeros_like(x)
        ref.level_apply(0, x, y)
        residuals.append(y)

    def apply(h):
        out = []
        for r in residuals:
            z = torch.zeros_like(r)
            h.apply_preconditioner(r, z)
            z[nu:] -= (w @ z[nu:]) / w.sum()
            out.append(z)
        return out

    want = apply(ref)

    def error(**o):
        got = apply(handle(prob, smoother=smoother, precision=1, **o))
        return np.sqrt(np.mean([float((a - b).norm() / b.norm()) ** 2
                                for a, b in zip(got, want)]))

    assert error() <= 2.0 * error(cluster_from=0, cycle_kernel=1)

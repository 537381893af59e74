"""The stored coarse cycle where device memory is short: it takes a small share of what is
free, and a call that finds no room for its own vectors gives it back and runs without it."""
import numpy as np
import pytest

from fem_inputs import problems as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def B():
    from paper_1503_01287_gb300 import binding
    return binding


def fill_device(leave):
    """A buffer that leaves about `leave` bytes of the device free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def mixed(n):
    """Braess-Sarazin, FP32, FGMRES(300): 12^3 stores 7,000 unknowns in 190 MB, and its two
    Krylov bases take 150 and 74 MB."""
    prob = fp.mixed_elasticity_problem(n, nu=0.45, seed=4)
    h = B().setup_problem(prob, B().default_options(smoother=3, precision=1, gmres_restart=300))
    b = torch.from_numpy(np.ascontiguousarray(prob.rhs())).cuda()
    return h, b


def test_krylov_vectors_come_before_the_stored_cycle():
    small, sb = mixed(4)
    assert small.solve(sb, torch.zeros_like(sb), 1e-8, True).converged   # the kernels are loaded
    h, b = mixed(12)
    x = torch.zeros_like(b)
    r, z = torch.randn_like(b), torch.zeros_like(b)
    hog = fill_device(190 * MB)
    st = h.solve(b, x, 1e-8, True)
    del hog
    torch.cuda.empty_cache()
    assert st.converged and st.stored_from == 0
    ref, _ = mixed(12)
    y = torch.zeros_like(b)
    st = ref.solve(b, y, 1e-8, True)
    assert st.converged and st.stored_from == 2
    assert float((x - y).norm() / y.norm()) < 1e-6
    h.apply_preconditioner(r, z)
    ref.apply_preconditioner(r, y)
    assert float((z - y).norm() / y.norm()) < 200 * 2.0 ** -24


def test_stored_cycle_takes_a_small_share():
    hog = fill_device(4096 * MB)
    h, b = mixed(12)
    x = torch.zeros_like(b)
    st = h.solve(b, x, 1e-8, True)
    del hog
    assert st.converged and st.stored_from == 0
    h.free()
    torch.cuda.empty_cache()
    h, b = mixed(12)
    assert h.solve(b, x, 1e-8, True).stored_from == 2


def test_batched_solves_give_the_stored_cycles_back():
    # a stored level of 5,202 unknowns (108 MB) each; a problem's batch vectors take 62 MB
    probs = [fp.elasticity_problem(11, seed=k) for k in range(3)]
    small = fp.elasticity_problem(4, seed=1)
    rng = np.random.default_rng(3)

    def setup(ps):
        hs, bs = [], []
        for p in ps:
            hs.append(B().setup_problem(p, B().default_options(precision=1)))
            b = rng.standard_normal((16, 3 * p.n_nodes))
            b[:, np.repeat((p.tags & fp.TAG_DIRICHLET) != 0, 3)] = 0.0
            bs.append(torch.from_numpy(b).cuda())
        return hs, bs, [torch.zeros_like(b) for b in bs]

    assert B().solve_batched(*setup([small]), 16, 1e-8)[0] == 0     # the kernels are loaded
    hs, bs, xs = setup(probs)
    hog = fill_device(150 * MB)
    rc, st = B().solve_batched(hs, bs, xs, 16, 1e-8)
    del hog
    assert rc == 0
    torch.cuda.empty_cache()
    ref, _, ys = setup(probs)
    rc, sr = B().solve_batched(ref, bs, ys, 16, 1e-8)
    assert rc == 0
    for x, y, a, c in zip(xs, ys, st, sr):
        assert abs(a.iterations - c.iterations) <= 1
        assert float((x - y).norm() / y.norm()) < 1e-6

"""Colour kernels under programmatic dependent launch: they are resident while the colours
before them still write x, so they read x through L2 and never by the non-coherent path.
The rule is checked on the source; batched solves of several problems side by side are
repeated bit for bit."""
import os
import re

import numpy as np
import pytest

from fem_inputs import problems as fp

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_01287_gb300", "csrc")


def dependent_kernels():
    """(name, body) of every kernel that waits on the grids before it."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as src:
            text = re.sub(r"//[^\n]*", "", src.read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            start = text.index("{", m.end())
            depth, end = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            if "griddepcontrol.wait" in text[start:end]:
                out.append((m.group(1), text[start:end]))
    return out


def test_dependent_kernels_read_x_through_l2():
    kernels = dependent_kernels()
    assert {"k_gs_pdl", "k_gs_m_pdl", "k_gs_m_staged"} <= {k for k, _ in kernels}
    for name, body in kernels:
        bad = re.findall(r"\b(?:ld3c?|ldg|__ldg|VL<false>::\w+)\s*\(\s*x4?\b[^;]*;", body)
        assert not bad, (name, bad)


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tile", [(1, -1), (1, 1), (1, 6), (0, -1), (0, 5)])
def test_batched_solves_repeat_bit_for_bit(precision, tile):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1503_01287_gb300 import binding as B
    probs = [fp.elasticity_problem(s, seed=k, nu=0.35)
             for k, s in enumerate([(9, 7, 8), (6, 11, 5), 8, (5, 5, 12)])]
    rng = np.random.default_rng(3)
    hs, bs, xs = [], [], []
    for p in probs:
        b = rng.standard_normal((16, 3 * p.n_nodes))
        b[:, np.repeat((p.tags & fp.TAG_DIRICHLET) != 0, 3)] = 0.0
        # the SpMM tile is timed once a handle, so one handle serves all repeats
        hs.append(B.setup_problem(p, B.default_options(precision=precision, batch_tile=tile)))
        bs.append(torch.from_numpy(b).cuda())
        xs.append(torch.zeros_like(bs[-1]))
    first = None
    for _ in range(4):
        rc, st = B.solve_batched(hs, bs, xs, 16, 1e-9)
        assert rc == 0
        now = [x.clone() for x in xs] + [torch.tensor([s.iterations for s in st])]
        if first is None:
            first = now
        assert all(torch.equal(a, b) for a, b in zip(first, now))

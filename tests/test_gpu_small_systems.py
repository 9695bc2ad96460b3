"""The scatter of small systems (one row per warp) overlaps the end of the cell
kernel whose matrices it reads. Assemblies in a row that share the scratch, with
nothing waited for in between, and the same as a captured CUDA graph (where the
overlap is a programmatic edge) give the bits of assemblies that are waited for
one by one. No tolerance: the same kernels run on the same inputs."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from metrics import TOL, row_scaled_error, vec_error
from paper_1708_01773_gb300 import build, feasm, inputs

pytestmark = pytest.mark.gpu
N = 12  # assemblies in a row


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    feasm.lib()


@pytest.mark.parametrize("order, problem, shape, prec", [
    (1, 0, (3, 3, 3), "fp32"), (1, 0, (20, 21, 19), "fp64"), (1, 1, (16, 16, 15), "bf16"), (1, 1, (5, 4, 3), "fp64"),
    (2, 1, (4, 4, 3), "fp32"), (2, 0, (7, 6, 5), "fp64"), (3, 0, (3, 4, 3), "bf16"), (3, 1, (3, 2, 2), "fp64"),
])
def test_overlapped_scatter_in_a_row_and_captured(order, problem, shape, prec):
    prob = inputs.small_problem(shape, order, problem, seed=300 + order)
    sp = feasm.FESpace(prob)
    rng = np.random.default_rng(301)
    coefs = [torch.tensor(prob.coef * rng.uniform(0.5, 2.0, prob.coef.size), device="cuda") for _ in range(N)]
    one_by_one = []
    for c in coefs:
        one_by_one.append(sp.assemble(c, prec=prec))
        torch.cuda.synchronize()
    rp, col, val, rhs = oracle.assemble_csr(dataclasses.replace(prob, coef=coefs[-1].cpu().numpy()))
    assert row_scaled_error(rp, col, one_by_one[-1][0].cpu().numpy(), val) <= TOL[prec]
    assert vec_error(one_by_one[-1][1].cpu().numpy(), rhs) <= 1e-12
    out = [tuple(torch.full_like(t, np.nan) for t in one_by_one[0]) for _ in coefs]
    torch.cuda.synchronize()
    for _ in range(4):
        for c, (v, r) in zip(coefs, out):
            sp.assemble(c, v, r, prec=prec)
    torch.cuda.synchronize()
    for got, want in zip(out, one_by_one):
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])

    coef = coefs[0].clone()
    v, r = (torch.full_like(t, np.nan) for t in one_by_one[0])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):  # warm-up outside the capture
        sp.assemble(coef, v, r, prec=prec, stream=side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sp.assemble(coef, v, r, prec=prec, stream=torch.cuda.current_stream())
    for c, (want_v, want_r) in zip(coefs, one_by_one):
        coef.copy_(c)
        graph.replay()
        got_v, got_r = v.clone(), r.clone()
        torch.cuda.synchronize()
        assert torch.equal(got_v, want_v) and torch.equal(got_r, want_r)
    assert sp.status() == 0
    sp.close()


def shapes_around(rows):
    """The Q1 elasticity bricks of nearly equal sides with the most rows up to `rows` and the fewest above."""
    sizes = sorted((3 * (a + 1) * (b + 1) * (c + 1), (a, b, c)) for a in range(16, 40) for b in range(a, a + 3)
                   for c in range(b, b + 3))
    return [s for s in sizes if s[0] <= rows][-1][1], [s for s in sizes if s[0] > rows][0][1]


@pytest.mark.parametrize("above", [False, True])
def test_node_rows_on_both_sides_of_the_rule(above):
    """Q1 elasticity, whose larger systems take the three rows of a node together, at 320 rows per SM."""
    shape = shapes_around(320 * torch.cuda.get_device_properties(0).multi_processor_count)[above]
    prob = inputs.small_problem(shape, 1, 1, seed=302)
    rp, col, val, rhs = oracle.assemble_csr(prob)
    sp = feasm.FESpace(prob)
    coef = torch.tensor(prob.coef, device="cuda")
    for prec in ("fp32", "fp64", "bf16"):
        v, r = sp.assemble(coef, prec=prec)
        torch.cuda.synchronize()
        assert row_scaled_error(rp, col, v.cpu().numpy(), val) <= TOL[prec]
        assert vec_error(r.cpu().numpy(), rhs) <= 1e-12
    sp.close()

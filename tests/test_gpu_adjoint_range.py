"""The FP64 adjoint on Q1 cells over the range of u and of the mesh's unit. The
cell energies scale as u^2 h, and powers of two scale every intermediate value
exactly, so a scaled run must give the scaled energies of the unscaled one, which
the oracle checks to 1e-12; both forms of the kernel keep that bound, hence 2e-12
between two runs."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from metrics import vec_error
from paper_1708_01773_gb300 import build, feasm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    feasm.lib()


def energies(prob, u):
    sp = feasm.FESpace(prob)
    c = torch.full((1,), np.nan, dtype=torch.float64, device="cuda")
    g = sp.adjoint(torch.tensor(u, device="cuda"), torch.tensor(prob.coef, device="cuda"), 1.0, compliance=c, prec="fp64")
    torch.cuda.synchronize()
    status = sp.status()
    sp.close()
    return g.cpu().numpy(), float(c), status


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("u_exp, h_exp", [
    (-300, 0), (300, 0), (-490, 0), (490, 0), (-440, 0), (440, 0),  # u at and beyond the line between the two forms
    (0, -300), (0, 300), (0, -215), (0, 215), (-100, -200), (100, 200), (300, -300), (-300, 300), (-200, -310),
    (200, 310),
])
def test_energies_over_the_range(problem, u_exp, h_exp):
    prob = inputs.small_problem((5, 4, 3), 1, problem, seed=930)
    sp = feasm.FESpace(prob)
    u = inputs.unit_rms_field(sp.n_dofs, 9)
    dofs = sp.cell_dofs()
    sp.close()
    u[dofs[7]] = 0.0   # one cell where nothing moves
    ref, c_ref, _ = energies(prob, u)
    assert vec_error(ref, oracle.cell_energies(prob, u, dofs)) <= 1e-12 and ref[7] == 0.0
    m = prob.mesh
    scaled = dataclasses.replace(prob, mesh=inputs.Mesh(np.ldexp(m.coords, h_exp), m.cell_vertices, m.shape, m.extent))
    g, c, status = energies(scaled, np.ldexp(u, u_exp))
    assert status == 0 and g[7] == 0.0
    assert vec_error(np.ldexp(g, -2 * u_exp - h_exp), ref) <= 2e-12
    assert abs(np.ldexp(c, -2 * u_exp - h_exp) - c_ref) <= 2e-12 * abs(c_ref)


@pytest.mark.parametrize("problem", [0, 1])
def test_one_node_out_of_range_changes_its_cells_only(problem):
    prob = inputs.small_problem((5, 4, 3), 1, problem, seed=931)
    sp = feasm.FESpace(prob)
    u = inputs.unit_rms_field(sp.n_dofs, 10)
    dofs = sp.cell_dofs()
    sp.close()
    ref, _, _ = energies(prob, u)
    for value in (np.nan, np.inf, 2.0**480):
        v = u.copy()
        v[dofs[30][0]] = value
        g, _, _ = energies(prob, v)
        hit = (dofs == dofs[30][0]).any(axis=1)
        assert np.array_equal(g[~hit], ref[~hit])
        if value == 2.0**480:
            assert vec_error(np.ldexp(g[hit], -960), np.ldexp(oracle.cell_energies(prob, np.ldexp(v, -100), dofs)[hit], -760)) <= 1e-12
        else:
            assert not np.isfinite(g[hit]).any()

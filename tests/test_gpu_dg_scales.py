"""IP-DG, FP64 form: facets between cells of very different thickness, and cells
whose facet weights leave the range of the fixed-point products."""
import numpy as np
import pytest
import torch

from dg_reference import dg_values
from metrics import row_scaled_error
from paper_1708_01773_gb300 import build, feasm, inputs

pytestmark = pytest.mark.gpu
# 64 units of 2^-52 per entry, relative to the row's largest: about 30 roundings of
# the point's geometry, as many in sums over at most 16 points. A weight in 36
# bits would show as 2^-37. The reference is in extended precision: the FP64 one
# forms Jacobians from positions, 2e-12 (ratio 2^10) and 4e-8 (2^24) off here.
TOL = 64 * 2.0**-52


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    feasm.lib()


def layers(order, z, seed=940):
    """A 3 x 2 brick whose vertex layers lie at the given heights, distorted in x and y only."""
    mesh = inputs.small_problem((3, 2, len(z) - 1), order, 0, seed=seed, alpha=0.0).mesh
    rng = np.random.default_rng(seed)
    coords = np.array(mesh.coords)
    level = np.rint(coords[:, 2] * (len(z) - 1)).astype(int)
    inner = (coords[:, :2] > 1e-9).all(axis=1) & (coords[:, :2] < 1 - 1e-9).all(axis=1)
    shift = 0.15 * rng.uniform(-1, 1, (coords.shape[0], 2)) / np.array([3, 2])
    coords[inner, :2] += np.round(shift[inner] * 2**20) / 2**20
    coords[:, 2] = np.asarray(z, dtype=np.float64)[level]
    return inputs.Mesh(coords, mesh.cell_vertices, mesh.shape, mesh.extent)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("scrambled", [False, True])
@pytest.mark.parametrize("ratio", [10, 24])
def test_graded_layers(order, scrambled, ratio):
    """Layers of thickness 1, 2^-ratio, 1: every row, among them those of the thick cells' nodes off the face."""
    t = 2.0**-ratio
    mesh = layers(order, [0.0, 1.0, 1.0 + t, 2.0 + t])
    if scrambled:
        mesh, _ = inputs.scramble(mesh, np.random.default_rng(5))
    g = feasm.DGSpace(mesh, order)
    for tau in (1.0, -0.7):
        rp, col = (x.cpu().numpy() for x in g.pattern())
        val = dg_values(mesh, order, tau, 12.0, g.facets(), rp, col)
        v, _ = g.assemble(tau, 12.0, 2.0, prec="fp64")
        torch.cuda.synchronize()
        assert row_scaled_error(rp, col, v.cpu().numpy(), val.astype(np.float64)) <= TOL
    g.close()


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("tau", [1.0, -0.7])
def test_weights_outside_the_fixed_point_range(order, tau):
    """Cells of thickness t = 2^-900: the weights through their faces are 2^900, those through their sides 2^-900. Up
    to parts t^2 of an entry the matrix is 1/t times a fixed one, which t = 2^-300 (in range) gives as well."""
    vals = {}
    for k in (300, 900):
        t = 2.0**-k
        g = feasm.DGSpace(layers(order, [0.0, t, 2 * t, 3 * t]), order)
        v, _ = g.assemble(tau, 12.0, 2.0, prec="fp64")
        rp, col = (x.cpu().numpy() for x in g.pattern())
        vals[k] = np.ldexp(v.cpu().numpy(), -k)
        if k == 300:
            ref = dg_values(layers(order, [0.0, t, 2 * t, 3 * t]), order, tau, 12.0, g.facets(), rp, col)
            ref = np.ldexp(ref, -300).astype(np.float64)
            assert row_scaled_error(rp, col, vals[k], ref) <= TOL
        g.close()
    assert np.isfinite(vals[900]).all() and row_scaled_error(rp, col, vals[900], ref) <= TOL


def test_nan_position_reaches_its_facets_only():
    mesh = layers(2, [0.0, 1.0, 2.0, 3.0])
    g = feasm.DGSpace(mesh, 2)
    want, _ = g.assemble(1.0, 12.0, 2.0, prec="fp64")
    g.close()
    coords = np.array(mesh.coords)
    coords[0] = np.nan  # a corner of cell 0
    g = feasm.DGSpace(inputs.Mesh(coords, mesh.cell_vertices, mesh.shape, mesh.extent), 2)
    got, _ = g.assemble(1.0, 12.0, 2.0, prec="fp64")
    rp, col = (x.cpu().numpy() for x in g.pattern())
    plus, minus, *_ = g.facets()
    g.close()
    got, want = got.cpu().numpy(), want.cpu().numpy()
    rows = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    near = np.isin(np.arange(mesh.n_cells), np.concatenate([[0], minus[plus == 0], plus[minus == 0]]))
    far = ~near[rows // 27] & ~near[col // 27]
    assert far.any() and np.array_equal(got[far], want[far]) and np.isnan(got).any()
    own = (rows // 27 == 0) & (col // 27 == 0)
    assert not np.isfinite(got[own]).any()

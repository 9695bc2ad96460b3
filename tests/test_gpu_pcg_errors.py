"""Loads and matrices for which the sums of the PCG of fe_compliance leave the
range of FP64: an error, never a result. FE_ERR_INVALID_ARG is what a diverged
solve and an indefinite matrix give."""
import numpy as np
import pytest
import torch

from paper_1708_01773_gb300 import build, feasm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    feasm.lib()


def clamped(shape, order=1, problem=1):
    prob = inputs.small_problem(shape, order, problem, seed=920, extent=(2.0, 1.0, 1.0))
    sp = feasm.FESpace(prob)
    return prob, sp.dirichlet(np.abs(sp.dof_points()[:, 0]) < 1e-12)


@pytest.mark.parametrize("shape", [(4, 2, 2), (38, 38, 38)])  # vectors in registers, in memory
@pytest.mark.parametrize("load, stiffness", [
    (540, 0),       # f.f overflows
    (500, -400),    # f.f near 2^1000: f.D^-1 f overflows
    (505, -8),      # the squares of the load are finite, p.A p or a later residual may not be
    (511, -20),
    (np.nan, 0),
    (np.inf, 0),
])
def test_sums_out_of_range_are_an_error(shape, load, stiffness):
    prob, dsys = clamped(shape)
    coef = torch.tensor(np.ldexp(prob.coef, stiffness), device="cuda")
    force = np.array([0.0, 0.0, load]) if not np.isfinite(load) else np.ldexp(prob.force, int(load))
    try:
        u, c, g, it, rel = dsys.compliance(coef, prec="fp64", rtol=1e-6, force=force)
    except feasm.FEError as e:
        assert e.code == -1  # FE_ERR_INVALID_ARG
    else:
        # every sum stayed in range: then the solution is the scaled one
        assert load in (505, 511) and rel <= 1e-6 and bool(torch.isfinite(u).all())
        w, _, _, _, _ = dsys.compliance(torch.tensor(prob.coef, device="cuda"), prec="fp64", rtol=1e-6)
        back = torch.tensor(float(stiffness - int(load)), dtype=torch.float64, device="cuda")
        # both meet rtol, cond(K) < 1e5 on these meshes
        assert float((torch.ldexp(u, back) - w).norm()) <= 2 * 1e-6 * 1e5 * float(w.norm())


def test_one_infinite_coefficient_is_an_error():
    prob, dsys = clamped((4, 2, 2))
    for bad in (np.inf, np.nan):
        coef = np.array(prob.coef)
        coef[5] = bad
        with pytest.raises(feasm.FEError) as ei:
            dsys.compliance(torch.tensor(coef, device="cuda"), prec="fp64", rtol=1e-6)
        assert ei.value.code == -1

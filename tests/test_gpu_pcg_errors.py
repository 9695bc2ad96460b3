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


@pytest.mark.parametrize("shape, order, problem", [((1, 1, 1), 1, 0), ((16, 17, 15), 1, 1), ((38, 38, 38), 1, 1),
                                                   ((10, 9, 9), 2, 1)])
def test_fewer_blocks_than_the_gpu_has(shape, order, problem):
    """Cooperative launches above max_blocks are answered with the runtime's error
    for a grid that does not fit. The residual is within the bound of the full
    grid's (1.1 rtol), and the number of blocks does not change the result:
    the partial sums belong to virtual blocks."""
    prob, dsys = clamped(shape, order, problem)
    coef = torch.tensor(prob.coef, device="cuda")
    vals, f = dsys.assemble(coef, None, prec="fp64")
    rp, col = dsys.pattern()
    label = torch.tensor(dsys.labels().astype(np.int64), device="cuda")
    rows = torch.repeat_interleave(torch.arange(dsys.n_free, device="cuda"), rp.diff())
    work = torch.empty(feasm.fe_compliance_work_size(dsys.handle), dtype=torch.float64, device="cuda")
    _, _, _, it_full, _ = dsys.compliance(coef, prec="fp64", rtol=1e-6)
    results = []
    for blocks in (1, 7, 75):
        u = torch.full((dsys.space.n_dofs,), np.nan, dtype=torch.float64, device="cuda")
        c = torch.empty(1, dtype=torch.float64, device="cuda")
        it, rel = feasm.fe_selftest_compliance(dsys.handle, coef, prob.force, feasm.PRECISIONS["fp64"], 1e-6, 20000,
                                               work, u, c, blocks)
        x = torch.zeros(dsys.n_free, dtype=torch.float64, device="cuda")
        x[label[label >= 0]] = u[label >= 0]
        r = f.clone().index_add_(0, rows, -vals * x[col.long()])
        assert rel <= 1e-6 and float(r.norm()) <= 1.1e-6 * float(f.norm())
        assert abs(it - it_full) <= 8  # one interval between checks: the sums' order differs
        results.append((it, rel, u, c))
    if dsys.n_free > 32:  # (fewer rows make one virtual block: the full grid, vectors in registers)
        for it, rel, u, c in results[1:]:
            assert (it, rel) == results[0][:2] and torch.equal(u, results[0][2]) and torch.equal(c, results[0][3])

"""FP64 form: the operator annihilates translations up to its roundings, also on
the boundary, where what a bias of the contraction's operands leaves does not
cancel between the cells around a node (and where the sum of all entries, second
order in such a bias, does not see it).

For each face of the brick the entries of the rows (node on the face, normal
component) in the columns of that component are summed, in integers (wrap-around
is harmless, the sum is small). Independent roundings of standard deviation at
most 2^-53 / sqrt(3) of their entry stay within 7.5 times that of the entries'
2-norm (6 standard deviations, a quarter more for the cells' own roundings); the
conversion's ties move an entry by 2^-61 of itself on average. Operands rounded
up at every tie (a quarter unit of 2^-59 on average) leave up to 1.7 times the bound."""
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


@pytest.mark.parametrize("order, problem, n", [(1, 1, 40), (1, 0, 48), (2, 1, 16), (2, 0, 24)])
def test_translations_on_the_faces(order, problem, n):
    prob = inputs.small_problem((n, n, n), order, problem, seed=950)
    sp = feasm.FESpace(prob)
    v, _ = sp.assemble(torch.tensor(prob.coef, device="cuda"), prec="fp64")
    rp, col = sp.pattern()
    nc = 3 if problem == 1 else 1
    pos = sp.dof_points()
    comp = np.zeros(sp.n_dofs, dtype=np.int64)   # component of each DOF, from the cells' local order (component-major)
    cd = sp.cell_dofs()
    nb = cd.shape[1] // nc
    for k in range(nc):
        comp[cd[:, k * nb:(k + 1) * nb].ravel()] = k
    comp = torch.tensor(comp, device="cuda")
    rows = torch.repeat_interleave(torch.arange(sp.n_dofs, device="cuda"), rp.diff())
    k = 61 - int(np.ceil(np.log2(float(v.abs().max()))))
    scaled = torch.round(torch.ldexp(v, torch.tensor(float(k), dtype=torch.float64, device="cuda"))).to(torch.int64)
    for axis in range(3):
        for side in (0.0, 1.0):
            face = torch.tensor(np.abs(pos[:, axis] - side) < 1e-9, device="cuda")
            want = axis if nc == 3 else 0
            take = face[rows] & (comp[rows] == want) & (comp[col.long()] == want)
            total = float(scaled[take].sum()) * 2.0 ** -k
            bound = 7.5 * 2.0**-53 / 3**0.5 * float(v[take].norm()) + 2.0**-61 * float(v[take].abs().sum())
            print(order, problem, axis, side, total, bound, total / bound)
            assert abs(total) <= bound
    sp.close()


@pytest.mark.parametrize("order, problem, n", [(1, 0, 64), (1, 1, 48), (2, 0, 24), (2, 1, 16)])
@pytest.mark.parametrize("contrast", ["2^-8 or 1", "2^-40 or 1", "2^-16 to 1"])
def test_sum_of_all_entries_with_coefficient_contrast(order, problem, n, contrast):
    """The scatter's sums lose bits only where their terms differ by more than 2^5, as they do between cells of very
    different coefficients. All entries together cancel; the bound is the one above. What is cut off (0.4 units of 2^-57
    of an entry and addition on average) must cancel with them: cut off downwards it is 3.8 times the bound."""
    prob = inputs.small_problem((n, n, n), order, problem, seed=92)
    rng = np.random.default_rng(1)
    cells = prob.coef.size
    coef = {"2^-8 or 1": np.where(rng.random(cells) < 0.5, 1.0, 2.0**-8),
            "2^-40 or 1": np.where(rng.random(cells) < 0.5, 1.0, 2.0**-40),
            "2^-16 to 1": 2.0 ** rng.uniform(-16, 0, cells)}[contrast]
    sp = feasm.FESpace(prob)
    v, _ = sp.assemble(torch.tensor(coef, device="cuda"), prec="fp64")
    k = 61 - int(np.ceil(np.log2(float(v.abs().max()))))
    scaled = torch.round(torch.ldexp(v, torch.tensor(float(k), dtype=torch.float64, device="cuda"))).to(torch.int64)
    total = float(scaled.sum()) * 2.0 ** -k
    bound = 7.5 * 2.0**-53 / 3**0.5 * float(v.norm()) + 2.0**-61 * float(v.abs().sum())
    print(order, problem, contrast, total, bound, total / bound)
    assert abs(total) <= bound
    sp.close()

"""Iteration and subset counts of the reconstructions: none or negative ones
return the start image, as a loop over them does, and only whole numbers are
taken."""
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plan():
    from paper_1607_06170_gb300 import build, psf as P

    build.build()
    w = I.workload("RING3D_SMALL")
    s, t, im, ls = w["scanner"], w["table"], w["image"], w["lors"]
    T, eta = P.response_build(s, t)
    W = P.bin_spread_classes(s, t, T, eta, ls, P.lor_set_classes(s, ls), *w["window"])
    idx, wk = P.spread_topn(W, *w["window"], 5)
    rows = P.sysmat_rows_set(s, im, ls)
    M = P.Matrix(*rows, im["nx"] * im["ny"] * im["nz"])
    return M.set_spread_topn(s, ls, *w["window"], idx, wk).build_sparse_adjoint()


def _start(M, x0):
    sens = M.sensitivity()
    return (sens >= 1e-12 * sens.max()).float() * (sens > 0) if x0 is None else x0


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("iters", [-3, -1, 0])
def test_mlem_without_iterations(plan, iters, given):
    from paper_1607_06170_gb300.torch_api import mlem

    y = torch.ones(plan.n_rows, device="cuda")
    x0 = torch.rand(plan.n_cols, device="cuda") if given else None
    assert torch.equal(mlem(plan, y, iters, x0), _start(plan, x0))


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("iters,subsets", [(-2, 2), (0, 2), (1, -1), (0, -4)])
def test_osem_without_iterations(plan, iters, subsets, given):
    from paper_1607_06170_gb300.torch_api import listmode_osem

    rows = torch.arange(0, plan.n_rows, 977, device="cuda")
    x0 = torch.rand(plan.n_cols, device="cuda") if given else None
    assert torch.equal(listmode_osem(plan, rows, subsets, iters, x0), _start(plan, x0))


def test_counts_are_whole_numbers(plan):
    from paper_1607_06170_gb300.torch_api import listmode_osem, mlem

    y = torch.ones(plan.n_rows, device="cuda")
    rows = torch.arange(0, plan.n_rows, 977, device="cuda")
    for call in (lambda: mlem(plan, y, 1.5), lambda: listmode_osem(plan, rows, 2, 1.5),
                 lambda: listmode_osem(plan, rows, 2.5, 1)):
        with pytest.raises(TypeError):
            call()

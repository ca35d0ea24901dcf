"""A plan whose launches were tuned, given other spreads or another grid later:
every projection still runs, and gives what a fresh plan of that state gives."""
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


@pytest.fixture(scope="module")
def ring(P):
    """Half of the 3D ring: large enough that the pair-streamed back-projection is
    the faster one by far, so that tuning takes it."""
    w = I.workload("RING3D")
    s = dict(w["scanner"], n_block_rings=2)
    ls, win = dict(fan_half=60, max_ring_diff=15), (3, 2)
    im = I.image(160, 160, 52, 0.8, 0.8, 1.1)
    T, eta = P.response_build(s, w["table"])
    W = P.bin_spread_classes(s, w["table"], T, eta, ls, P.lor_set_classes(s, ls), *win)
    return s, ls, im, win, W, P.spread_topn(W, *win, 5), P.sysmat_rows_set(s, im, ls)


def _kernels(P, f):
    P.timing_enable(True)
    out = f()
    ran = set(P.timing_read())
    P.timing_enable(False)
    return out, ran


def _all(M, x, y):
    return (M.forward(x), M.back(y), *M.back_sens(y), M.sensitivity())


def _agree(got, want, what):
    for g, o in zip(got, want):
        # sums of the same positive FP32 products in another order
        assert_close(g.cpu(), o.cpu(), 5e-5, 1e-6 * float(o.abs().max()), what)


@pytest.mark.parametrize("then", ["topn", "grid without a pair form", "grid of long rows"])
def test_tuned_plan_changed_later(P, ring, then):
    from paper_1607_06170_gb300.torch_api import listmode_osem

    s, ls, im, win, W, (idx, wk), rows = ring
    nv = im["nx"] * im["ny"] * im["nz"]
    x, y = torch.rand(nv, device="cuda"), torch.rand(rows[0].numel() - 1, device="cuda")
    M = P.Matrix(*rows, nv).set_spread(s, ls, *win, W).set_image(im)
    M.autotune()
    before, ran = _kernels(P, lambda: _all(M, x, y))
    assert "csr_back_single_kernel" in ran  # the choice that the change makes stale
    R = P.Matrix(*rows, nv).set_launch(0)
    if then == "topn":
        M.set_spread_topn(s, ls, *win, idx, wk)
        R.set_spread_topn(s, ls, *win, idx, wk)
        ev = torch.arange(0, M.n_rows, 401, device="cuda")
        got = listmode_osem(M, ev, 2, sparse_adjoint=False)
        _agree([got], [listmode_osem(R, ev, 2, sparse_adjoint=False)], "OSEM image")
    else:
        R.set_spread(s, ls, *win, W)
        M.set_image(I.image(1, 1, nv, 1.0, 1.0, 1.0) if "without" in then else
                    I.image(51200, 26, 1, 1.0, 1.0, 1.0))
    _agree(_all(M, x, y), _all(R, x, y), then)
    M.set_spread(s, ls, *win, W).set_image(im)  # and back: the tuned choice again
    after, ran = _kernels(P, lambda: _all(M, x, y))
    assert "csr_back_single_kernel" in ran
    _agree(after, before, "restored")
    M.check()


def test_plan_tuned_before_its_image(P, ring):
    """Tuned without a grid (or with truncated spreads), the plan still takes the
    pair form where it fits once the grid (the full spreads) is there."""
    s, ls, im, win, W, (idx, wk), rows = ring
    nv = im["nx"] * im["ny"] * im["nz"]
    x, y = torch.rand(nv, device="cuda"), torch.rand(rows[0].numel() - 1, device="cuda")
    R = P.Matrix(*rows, nv).set_spread(s, ls, *win, W).set_launch(0)
    want = _all(R, x, y)
    M = P.Matrix(*rows, nv).set_spread(s, ls, *win, W)
    M.autotune()
    M.set_image(im)
    K = P.Matrix(*rows, nv).set_spread_topn(s, ls, *win, idx, wk).set_image(im)
    K.autotune()
    K.set_spread(s, ls, *win, W)
    for plan in (M, K):
        got, ran = _kernels(P, lambda: _all(plan, x, y))
        assert {"csr_fwd_patch_kernel", "csr_back_single_kernel"} <= ran
        _agree(got, want, "tuned before")

"""The reconstructions over objects other than a psf.Matrix itself: what they
need is the object's own forward, back, back_sens and sensitivity (CPU: the EM
steps' kernels stand in as torch code)."""
import pytest
import torch

from paper_1607_06170_gb300 import psf, torch_api

N, V = 23, 11
A = torch.rand((N, V), generator=torch.Generator().manual_seed(5)) + 0.1
GAIN = torch.linspace(0.5, 2.0, N)  # a normalisation that the object applies


class Projections:
    n_rows, n_cols, topn = N, V, 0

    def __init__(self):
        self.calls = []

    def forward(self, x, out=None):
        self.calls.append("forward")
        y = GAIN * (A @ x)
        return y if out is None else out.copy_(y)

    def forward_masked(self, x, mask, out=None):
        self.calls.append("forward_masked")
        y = torch.where(mask != 0, GAIN * (A @ x), 0.0)
        return y if out is None else out.copy_(y)

    def back(self, y, out=None):
        self.calls.append("back")
        x = A.T @ (GAIN * y)
        return x if out is None else out.copy_(x)

    def back_sens(self, y, out=None, sens=None):
        self.calls.append("back_sens")
        return A.T @ (GAIN * y), A.T @ GAIN

    def sensitivity(self, out=None, device="cpu"):
        self.calls.append("sensitivity")
        return A.T @ GAIN


class Derived(Projections, psf.Matrix):
    """A psf.Matrix with projections of its own."""

    _h = None

    def build_sparse_adjoint(self):
        return self


def _patched():
    """A psf.Matrix whose instance carries its own projections."""
    own, M = Projections(), psf.Matrix.__new__(psf.Matrix)
    M._h = None
    for k in ("forward", "forward_masked", "back", "back_sens", "sensitivity", "n_rows", "n_cols",
              "topn", "calls"):
        setattr(M, k, getattr(own, k))
    M.build_sparse_adjoint = lambda: M
    return M


@pytest.fixture(autouse=True)
def steps(monkeypatch):
    def ratio(y, yhat, out=None):
        r = torch.where(yhat > 0, y / yhat, 0.0)
        return r if out is None else out.copy_(r)

    def update(x, bp, sens, floor):
        return x.copy_(torch.where((sens >= floor) & (sens > 0), x * bp / sens, 0.0))

    def histogram(rows, n_rows, weight=1.0, out=None):
        h = weight * torch.bincount(rows[(rows >= 0) & (rows < n_rows)], minlength=n_rows).float()
        return h if out is None else out.copy_(h)

    monkeypatch.setattr(psf, "em_ratio", ratio)
    monkeypatch.setattr(psf, "em_update", update)
    monkeypatch.setattr(psf, "histogram", histogram)


def _em(y, x, weight=1.0):
    return x * (A.T @ (GAIN * torch.where(y != 0, y / (GAIN * (A @ x)), 0.0))) / (A.T @ GAIN)


@pytest.mark.parametrize("make", [Projections, Derived, _patched])
@pytest.mark.parametrize("start", ["nothing", "sens", "x0", "both"])
@pytest.mark.parametrize("iters", [0, 1, 3])
def test_mlem_calls_the_objects_projections(make, start, iters):
    M = make()
    y = GAIN * (A @ torch.linspace(1.0, 2.0, V))
    x0 = torch.linspace(0.5, 1.5, V)
    got = torch_api.mlem(M, y, iters, x0 if start in ("x0", "both") else None,
                         A.T @ GAIN if start in ("sens", "both") else None)
    want = x0 if start in ("x0", "both") else torch.ones(V)
    for _ in range(iters):
        want = _em(y, want)
    # three iterations of FP32 sums of at most 23 terms
    torch.testing.assert_close(got, want, rtol=3e-5, atol=0)
    assert M.calls.count("forward") == iters


@pytest.mark.parametrize("make", [Projections, Derived, _patched])
@pytest.mark.parametrize("topn", [0, 5])
def test_osem_calls_the_objects_projections(make, topn):
    M = make()
    M.topn = topn
    M.build_sparse_adjoint = lambda: M
    M.n_rows = 640  # subsets of at most a sixteenth of the rows
    rows = torch.arange(60) % N

    def masked(x, mask, out=None):
        return out.copy_(torch.cat([Projections.forward_masked(M, x, mask[:N]),
                                    torch.zeros(640 - N)]))

    M.forward_masked = masked
    M.back = lambda y, out=None: out.copy_(Projections.back(M, y[:N]))
    got = torch_api.listmode_osem(M, rows, 2, 1, sens=A.T @ GAIN)
    want = torch.ones(V)
    for part in (rows[:30], rows[30:]):
        want = _em(2.0 * torch.bincount(part, minlength=N).float(), want)
    torch.testing.assert_close(got, want, rtol=3e-5, atol=0)
    assert M.calls.count("back") == 2

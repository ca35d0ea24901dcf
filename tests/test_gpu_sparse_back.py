"""psf_back of a pair-streamed plan when most LOR values are 0: past the rows
without one on large plans, streamed otherwise, the same image either way."""
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


def _plans(P, fan, dtype):
    w = I.workload("RING3D")
    s = dict(w["scanner"], n_block_rings=2)
    ls, win = dict(fan_half=fan, max_ring_diff=15), (1, 0)
    im = I.image(60, 72, 26, 2.0, 2.0, 2.2)
    T, eta = P.response_build(s, w["table"])
    W = P.bin_spread_classes(s, w["table"], T, eta, ls, P.lor_set_classes(s, ls), *win)
    rows = P.sysmat_rows_set_typed(s, im, ls, dtype)
    make = lambda: P.Matrix(*rows[:3], 60 * 72 * 26, row_scale=rows[3]).set_spread(s, ls, *win, W)
    return make().set_image(im), make().set_launch(0), rows


def _back(P, M, y):
    P.timing_enable(True)
    x = M.back(y)
    ms = {k: v[1] for k, v in P.timing_read().items()}
    P.timing_enable(False)
    return x, ms


def _streamed(ms):
    """Which of the two did the work: the other returns at once."""
    return ms["csr_back_single_kernel"] > ms["csr_back_wq_kernel"]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("fan", [12, 17])  # 2,207,400 and 3,090,360 rows
def test_back_by_density(P, fan, dtype, tuned):
    M, R, rows = _plans(P, fan, dtype)
    assert M.n_rows >= 1 << 21
    if tuned:
        M.autotune()
    n = M.n_rows
    g = torch.Generator(device="cuda").manual_seed(fan)
    dense = torch.rand(n, generator=g, device="cuda")
    keep = torch.rand(n, generator=g, device="cuda")
    for share in (0.0, 1e-6, 1e-3, 0.1, 0.4, 0.5, 0.6, 0.9, 1.0):
        y = torch.where(keep < share, dense, 0.0)
        got, ran = _back(P, M, y)
        assert "sample_sparse_kernel" in ran or tuned
        if "sample_sparse_kernel" in ran and share in (0.0, 1e-6, 1.0):
            assert _streamed(ran) == (share == 1.0)
        want = R.back(y)
        # sums of the same positive products in another order: up to ~2e4 per voxel
        assert_close(got.cpu(), want.cpu(), 2e-5, 1e-6 * float(want.abs().max()) + 1e-30, str(share))
    # values only where a row has entries: the empty rows say nothing about the work
    y = (rows[0][1:] > rows[0][:-1]).float()
    got, ran = _back(P, M, y)
    assert "sample_sparse_kernel" not in ran or _streamed(ran)
    assert_close(got.cpu(), R.back(y).cpu(), 2e-5, 1e-6 * float(got.max()), "rows with entries")
    one = torch.zeros(n, device="cuda")
    one[n // 2 + 77] = 2.0  # its neighbours' row starts are a whole pair's away
    assert_close(_back(P, M, one)[0].cpu(), R.back(one).cpu(), 2e-5, 1e-30, "one event")
    M.check()


def test_small_plans_stream(P):
    M, R, _ = _plans(P, 11, "f32")  # 2,030,808 rows
    assert M.n_rows < 1 << 21
    y = torch.zeros(M.n_rows, device="cuda")
    y[::1001] = 1.0
    got, ran = _back(P, M, y)
    assert "csr_back_single_kernel" in ran and "sample_sparse_kernel" not in ran
    assert_close(got.cpu(), R.back(y).cpu(), 2e-5, 1e-30, "small plan")


def test_sparse_back_is_captured(P):
    """The choice is taken on the device: a captured back-projection follows the
    values of each replay."""
    M, R, _ = _plans(P, 12, "f32")
    y, out = torch.ones(M.n_rows, device="cuda"), torch.empty(M.n_cols, device="cuda")
    M.back(y, out=out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        M.back(y, out=out)
    for step in (1, 997, 2):
        y.zero_()
        y[::step] = 1.0
        graph.replay()
        torch.cuda.synchronize()
        want = R.back(y)
        assert_close(out.cpu(), want.cpu(), 2e-5, 1e-6 * float(want.max()), f"every {step}")

"""MLEM on stored rows on both sides of the line between the fused kernels and the
separate ones (four rows a warp), rows of no entry to several hundred."""
import numpy as np
import pytest
import torch

from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("over", [-38000, -1, 0, 1, 9000])
def test_mlem_by_row_count(over, dtype):
    from paper_1607_06170_gb300 import build, psf as P
    from paper_1607_06170_gb300.torch_api import mlem

    build.build()
    line = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 8 * 4
    n, nv = line + over, 3001
    rng = np.random.default_rng(n)
    length = rng.choice([0, 1, 31, 33, 127, 128, 129, 160, 257, 300], n)
    ptr = torch.from_numpy(np.concatenate([[0], np.cumsum(length)])).cuda()
    nnz = int(length.sum())
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), ptr[1:] - ptr[:-1])
    col = ((torch.arange(nnz, device="cuda") - ptr[row]) * 7 + row * 13) % nv  # distinct in a row
    val = torch.rand(nnz, device="cuda") + 0.5
    scale = None
    if dtype == "bf16":
        val, scale = val.bfloat16(), torch.rand(n, device="cuda") + 0.5
    M = P.Matrix(ptr, col.int().contiguous(), val, nv, row_scale=scale)
    y = M.forward(torch.rand(nv, device="cuda") + 0.5)
    y[torch.rand(n, device="cuda") < 0.3] = 0.0
    sens = M.sensitivity()
    floor = 1e-12 * float(sens.max())
    for given in (None, sens):
        P.timing_enable(True)
        got = mlem(M, y, 3, None, given)
        ran = set(P.timing_read())
        P.timing_enable(False)
        # (a first iteration from ones takes the fused kernels at any size)
        assert ("mlem_ratio_kernel" in ran) == (n <= line or given is None)
        assert ("csr_fwd_kernel" in ran) == (n > line)
        x = torch.ones_like(sens)
        P.em_update(x, sens, sens, floor)
        for _ in range(3):
            P.em_update(x, M.back(P.em_ratio(y, M.forward(x))), sens, floor)
        # three iterations of FP32 sums of up to 2,500 terms in another order
        assert_close(got.cpu(), x.cpu(), 2e-5, 1e-6 * float(x.max()), "MLEM image")

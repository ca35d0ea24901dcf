"""MLEM calls that share one plan: with the sensitivity given, a plan without
spreads is only read, so reconstructions on several streams or from several
threads don't see each other.  And a plan without rows."""
import threading

import pytest
import torch

from paper_1607_06170_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


@pytest.fixture(scope="module", params=["stored", "bf16", "streaming launch", "bulk launch", "traced"])
def plan(P, request):
    w = I.workload("RING3D_SMALL")
    s, im, ls = w["scanner"], w["image"], w["lors"]
    if request.param == "traced":
        return P.Matrix.traced(s, im, ls)
    rows = P.sysmat_rows_set_typed(s, im, ls, "bf16" if request.param == "bf16" else "f32")
    M = P.Matrix(*rows[:3], im["nx"] * im["ny"] * im["nz"], row_scale=rows[3])
    return M.set_launch({"streaming launch": -1, "bulk launch": -2}.get(request.param, 0))


def _two(plan):
    """Data and sensitivities of two users: the second's has one voxel so bright
    that every other one is below its floor."""
    y = plan.forward(torch.rand(plan.n_cols, device="cuda") + 0.5)
    sens = plan.sensitivity()
    other = sens.clone()
    other[int(sens.argmax())] = 1e20
    return y, sens, other


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("how", ["streams", "threads"])
def test_two_reconstructions_with_one_plan(plan, how, given):
    from paper_1607_06170_gb300.torch_api import mlem

    y, *both = _two(plan)
    x0 = torch.rand(plan.n_cols, device="cuda") if given else None
    iters, calls = (40, 3), (1, 40)
    alone = [mlem(plan, y, k, x0, s) for k, s in zip(iters, both)]
    assert float(alone[0].max()) > 0 and int((alone[1] > 0).sum()) <= 1
    torch.cuda.synchronize()
    streams, got, errors = [torch.cuda.Stream() for _ in both], [[], []], []

    def user(i):
        try:
            with torch.cuda.stream(streams[i]):
                for _ in range(calls[i]):
                    got[i].append(mlem(plan, y, iters[i], x0, both[i]))
        except Exception as e:  # reaches the main thread
            errors.append(e)

    if how == "threads":
        users = [threading.Thread(target=user, args=(i,)) for i in (0, 1)]
        [u.start() for u in users]
        [u.join() for u in users]
    else:
        user(0), user(1)
    torch.cuda.synchronize()
    assert not errors
    for xs, want, k in zip(got, alone, iters):
        for x in xs:
            # k iterations of FP32 sums in another order, up to 7e-6 each
            torch.testing.assert_close(x, want, rtol=7e-6 * k + 1e-6, atol=1e-6 * float(want.max()))


@pytest.mark.parametrize("iters", [0, 2])
@pytest.mark.parametrize("start", ["nothing", "sens", "x0", "both"])
def test_plan_without_rows(P, iters, start):
    from paper_1607_06170_gb300.torch_api import mlem

    nv = 37
    M = P.Matrix(torch.zeros(1, dtype=torch.int64, device="cuda"),
                 torch.empty(0, dtype=torch.int32, device="cuda"), torch.empty(0, device="cuda"), nv)
    sens = torch.linspace(1e-14, 1.0, nv, device="cuda")
    x0 = torch.rand(nv, device="cuda") + 0.5
    with_x, with_s = start in ("x0", "both"), start in ("sens", "both")
    got = mlem(M, torch.empty(0, device="cuda"), iters, x0 if with_x else None, sens if with_s else None)
    want = x0 if with_x else (sens >= 1e-12).float() if with_s else torch.zeros(nv, device="cuda")
    assert torch.equal(got, want if iters == 0 else torch.zeros(nv, device="cuda"))

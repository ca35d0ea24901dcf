"""Totals of truncated windows in 64 bits where the terms nearly cancel or lie
far apart: the kept weights are the double computation's, rounded."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

WT, WA, E = 3, 3, 49


@pytest.fixture(scope="module")
def P():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


def _cancelling(rng, n):
    """Positive and negative entries that cancel to about 2^-27, the negative
    ones in every second piece of 77: multiples of 2^-40 below 2^11 in any
    partial sum, so that sums of doubles are exact in every order."""
    at = np.arange(E * E)
    minus, plus = at[at // 77 % 2 == 1], at[at // 77 % 2 == 0]
    w = np.zeros((n, E * E), dtype=np.float64)
    for row in w:
        a = rng.choice(np.arange(1 << 23, 1 << 24), len(minus), replace=False) * 2.0 ** -24
        plus_at = rng.permutation(plus)
        row[minus], row[plus_at[: len(a)]] = -rng.permutation(a), a
        row[plus_at[len(a):]] = rng.integers(1, 256, len(plus) - len(a)) * 2.0 ** -40
    return w


def _far_apart(rng, n):
    """A kept total of about 1e-24 in a window whose total is beyond -1e28: their
    quotient is no FP32 number, the weights are."""
    w = -rng.uniform(1e25, 2e25, size=(n, E * E))
    for row in w:
        row[rng.choice(E * E, 5, replace=False)] = rng.uniform(1e-24, 2e-24, 5)
    return w


@pytest.mark.parametrize("make,rtol", [(_cancelling, 0.0), (_far_apart, 2.0 ** -23)])
@pytest.mark.parametrize("N", [1, 5, 40])
def test_totals_in_64_bits(P, make, rtol, N):
    w = make(np.random.default_rng(N), 37).astype(np.float32)
    if make is _far_apart and N == 40:
        pytest.skip("entries that rank as 0 would be kept: one sign, no far quotient")
    idx, wk = P.spread_topn(torch.from_numpy(w.reshape(-1, E, E)).cuda(), WT, WA, N)
    idx, wk = idx.cpu().numpy().astype(np.int64), wk.cpu().numpy()
    sel = np.take_along_axis(w.astype(np.float64), idx, 1)
    best = np.sort(w, 1)[:, ::-1][:, :N]
    np.testing.assert_array_equal(sel, best)
    want = (sel * (w.astype(np.float64).sum(1) / sel.sum(1))[:, None]).astype(np.float32)
    np.testing.assert_allclose(wk, want, rtol=rtol, atol=0)

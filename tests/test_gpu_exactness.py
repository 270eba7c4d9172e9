"""Rounding of the sums over runs: results against float64 in units of their last place.

Run sums are carried in two floats, so a mean is rounded once: it lies within half an ulp of
the exact one, 0.05 ulp more for the quotient's residual, and 1e-12 for sums that cancel (two
floats of up to 4096 terms below 6 leave 4096 * 2^-48 * 300). Sums in one float miss that by
several ulp."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _ulp(ref):
    return np.spacing(np.abs(ref.astype(np.float32))).astype(np.float64)


def _means(x, g):
    cut = np.flatnonzero(np.r_[True, x[1:] != x[:-1]])
    cnt = np.diff(np.r_[cut, len(x)])
    return np.repeat(np.add.reduceat(g.astype(np.float64), cut) / cnt, cnt)


@pytest.mark.parametrize("n", [5, 33, 256, 700, 1024, 1025, 2048, 3000, 4096])
@pytest.mark.parametrize("top", [2, 40, 1000])
def test_backward_means(n, top):
    rng = np.random.default_rng(n + top)
    x = np.repeat(rng.normal(size=(6, n)), rng.integers(1, top + 1, n), axis=1)[:, :n].astype(np.float32)
    g = rng.normal(size=x.shape).astype(np.float32)
    gy = _lib.chain_prox_backward(torch.from_numpy(x).to(DEV), torch.from_numpy(g).to(DEV))[0].cpu().numpy()
    for a, b, got in zip(x, g, gy):
        ref = _means(a, b)
        assert (np.abs(got - ref) <= 0.55 * _ulp(ref) + 1e-12).all()

"""Gradients that are not finite in the backward kernels: a run's mean is what its float64 sum
over its length is, infinity of the same sign or NaN, wherever the run lies (inside a lane's
consecutive nodes, over several lanes, over several warps, beyond 4096 nodes), and every other
run is untouched."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [24, 900, 1500, 3000, 5000])
@pytest.mark.parametrize("length", [1, 3, 5, 40, 700])
def test_infinities_by_place(n, length):
    rng = np.random.default_rng(n + length)
    runs = -(-n // length)
    x = np.repeat(np.arange(runs), length)[:n].astype(np.float32)
    g = rng.normal(size=n).astype(np.float32)
    for r in range(0, runs, 3):  # +inf, -inf, NaN, inf - inf in turn, neighbours of them finite
        a, b = r * length, min(n, (r + 1) * length)
        g[a + (b - a) // 2] = [np.inf, -np.inf, np.nan, np.inf][r // 3 % 4]
        if r // 3 % 4 == 3:
            g[a] = -np.inf if b - a > 1 else np.inf
    with np.errstate(invalid="ignore"):
        ref = np.concatenate([np.full(min(n, (r + 1) * length) - r * length,
                                      g[r * length:(r + 1) * length].astype(np.float64).mean())
                              for r in range(runs)])
    xg, gg = (torch.from_numpy(a[None]).to(DEV) for a in (x, g))
    gy = _lib.chain_prox_backward(xg, gg)[0].cpu().numpy()[0]
    fine = np.isfinite(ref)
    assert np.array_equal(np.isnan(gy), np.isnan(ref))
    assert np.array_equal(gy[np.isinf(ref)], ref[np.isinf(ref)])
    # up to 700 terms N(0, 1), partial sums below 150: 700 additions of half an ulp of those
    assert np.abs(gy[fine] - ref[fine]).max(initial=0.0) <= 1e-5

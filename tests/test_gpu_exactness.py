"""Rounding of the sums over runs, against float64: they are carried in two floats, so that a
mean is rounded once."""
import numpy as np
import pytest
import torch

import oracle
from paper_1502_07770_gb300 import _lib, synth

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
    """Half an ulp, 0.05 for the quotient's residual, and 1e-12 for sums that cancel (two floats
    of up to 4096 terms below 6 leave 4096 * 2^-48 * 300). Sums in one float miss that by several
    ulp."""
    rng = np.random.default_rng(n + top)
    x = np.repeat(rng.normal(size=(6, n)), rng.integers(1, top + 1, n), axis=1)[:, :n].astype(np.float32)
    g = rng.normal(size=x.shape).astype(np.float32)
    gy = _lib.chain_prox_backward(torch.from_numpy(x).to(DEV), torch.from_numpy(g).to(DEV))[0].cpu().numpy()
    for a, b, got in zip(x, g, gy):
        ref = _means(a, b)
        assert (np.abs(got - ref) <= 0.55 * _ulp(ref) + 1e-12).all()


@pytest.mark.parametrize("n", [32, 100, 256, 700, 1023, 1024, 1025, 2048, 3000, 4096])
@pytest.mark.parametrize("edges", [False, True])
def test_chain_values(n, edges):
    """Of chains on the splitting kernel (rows from 20 nodes, columns from 32; shorter ones are the
    warp's dynamic program's). A value v rounded once is off by 2^e 2^-23 / sqrt(12) in the root mean square, 2^e <= v <
    2^(e+1): 2.3e-8 of v for mantissas spread evenly. 3.0e-8 of the norm leaves a third for the
    flows added to a run's end nodes. (The step-wise dynamic program's values: 3.2e-8, runs
    summed in one float 4.6e-8.)"""
    y = synth.chain_batch(12, n, seed0=n)
    w = np.random.default_rng(n).uniform(0.03, 0.3, y.shape).astype(np.float32) if edges else None
    ref = oracle.chain_solve_batch(y.ravel(), np.arange(13) * n, w=None if w is None else w.ravel(),
                                   lam=float(np.float32(0.2))).reshape(y.shape)
    g = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    x = _lib.chain_prox(g(y), g(w), lam=0.2).cpu().numpy()
    xc = _lib.chain_prox_columns(g(y.T), None if w is None else g(w.T), lam=0.2).cpu().numpy().T
    for got in (x, xc):
        assert np.linalg.norm(got - ref) <= 3.0e-8 * np.linalg.norm(ref)

"""Chains whose values lie near the ends of FP32's range, against the FP64 oracle: sums over a
chain would overflow, or weights count that are negligible beside ordinary values. The tolerance
is that of every chain kernel, 2e-5 on [0, 1] data, times the scale."""
import numpy as np
import pytest
import torch

import oracle
from paper_1502_07770_gb300 import _lib, synth

pytestmark = pytest.mark.gpu
TOL = 2e-5
DEV = "cuda:0"


def _gpu(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("scale", [1e37, 1e36, 1e32, 1e-27, 1e-29, 1e-36, 1e-38])
def test_scales(scale, edges):
    for n in (48, 300, 1024, 1500, 2600):
        y = synth.chain_batch(9, n, seed0=n).astype(np.float64)
        y[4] = 0.0  # a chain of zeros among them
        w = np.random.default_rng(n).uniform(0.02, 0.4, y.shape)
        ys, lam = (y * scale).astype(np.float32), np.float32(0.2 * scale)
        ws = (w * scale).astype(np.float32) if edges else None
        ref = oracle.chain_solve_batch(ys.ravel(), np.arange(10) * n, w=None if ws is None else ws.ravel(),
                                       lam=float(lam)).reshape(y.shape)
        x = _lib.chain_prox(_gpu(ys), _gpu(ws), lam=float(lam)).cpu().numpy()
        xc = _lib.chain_prox_columns(_gpu(ys.T), None if ws is None else _gpu(ws.T),
                                     lam=float(lam)).cpu().numpy().T
        for got in (x, xc):
            assert np.abs(got / scale - ref / scale).max() <= TOL, n


@pytest.mark.parametrize("n", [48, 300, 1024, 1500, 2600])
def test_nan_weights_go_to_the_dynamic_program(n):
    """A NaN weight is no cut: its chain gives what the warp's dynamic program (solve mode 0)
    makes of it, bit for bit; the entry at a chain's last node is not read. The other chains are
    untouched."""
    y = synth.chain_batch(9, n, seed0=n)
    w = np.full(y.shape, 0.2, np.float32)
    clean = _lib.chain_prox(_gpu(y), _gpu(w)).cpu().numpy()
    w[3, n // 3] = w[7, 0] = np.nan
    w[5, -1] = np.nan
    lib = _lib.load()
    try:
        _lib._check(lib.tv_set_coop_split(0))
        want = _lib.chain_prox(_gpu(y), _gpu(w)).cpu().numpy()
        wantc = _lib.chain_prox_columns(_gpu(y.T), _gpu(w.T)).cpu().numpy().T
    finally:
        _lib._check(lib.tv_set_coop_split(1))
    x = _lib.chain_prox(_gpu(y), _gpu(w)).cpu().numpy()
    xc = _lib.chain_prox_columns(_gpu(y.T), _gpu(w.T)).cpu().numpy().T
    for k in (3, 7):
        assert np.array_equal(x[k], want[k], equal_nan=True)
        assert np.array_equal(xc[k], wantc[k], equal_nan=True)
    rest = [k for k in range(9) if k not in (3, 7)]
    assert np.array_equal(x[rest], clean[rest]) and np.array_equal(xc[rest], clean[rest])

"""The threshold-splitting chain kernel (csrc/tv_split.cuh) against the FP64 oracle.

Tolerance 2e-5 as for every chain kernel on [0, 1] data. Lengths sit at the edges of what a
lane (4 to 32 nodes), a warp and 2, 4 or 8 warps hold, with the last lane part full, one node
long or empty; data that need few rounds (constant, fused), many (ramp, steps of every size),
and runs that cross lanes and warps.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1502_07770_gb300 import _lib, synth

pytestmark = pytest.mark.gpu
TOL = 2e-5
DEV = "cuda:0"
LENGTHS = [2, 3, 31, 32, 33, 128, 129, 256, 257, 384, 385, 511, 512, 513, 640, 641, 768, 769,
           1023, 1024, 1025, 1536, 1537, 2047, 2048, 2049, 3072, 3073, 4095, 4096]


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _data(n, rng):
    """Rows of one length: signals, a ramp, a constant, long plateaus, steps of all sizes."""
    y = synth.chain_batch(4, n, seed0=n)
    i = np.arange(n)
    more = [i / n, np.full(n, 0.3), np.repeat(rng.uniform(0, 1, -(-n // 300)), 300)[:n],
            np.sin(i * 0.02) + 0.02 * rng.normal(size=n), 2.0 ** -(i % 23)]
    return np.concatenate([y, np.stack(more).astype(np.float32)])


@pytest.mark.parametrize("n", LENGTHS)
def test_lengths_weights_rows_and_columns(n):
    rng = np.random.default_rng(n)
    y = _data(n, rng)
    B = len(y)
    w = rng.uniform(0.0, 0.4, size=y.shape).astype(np.float32)
    w[:, 5::17] = 0.0
    off = np.arange(B + 1) * n
    for lam, weights in ((0.2, None), (0.01, None), (3.0, None), (0.0, w)):
        ref = oracle.chain_solve_batch(y.ravel(), off, w=None if weights is None else weights.ravel(),
                                       lam=lam).reshape(y.shape)
        wr = None if weights is None else _gpu(weights)
        x = _lib.chain_prox(_gpu(y), wr, lam=lam).cpu().numpy()
        assert np.abs(x - ref).max() <= TOL, (lam, "rows")
        # fused neighbours are bitwise equal (the backward pass reads segments off x); an edge
        # of weight 0 fuses nothing
        fused = np.abs(np.diff(ref, axis=1)) < 1e-12
        if weights is not None:
            fused &= weights[:, :-1] > 0
        assert (fused <= (np.diff(x, axis=1) == 0)).mean() > 0.999
        wc = None if weights is None else _gpu(weights.T)
        xc = _lib.chain_prox_columns(_gpu(y.T), wc, lam=lam).cpu().numpy().T
        assert np.abs(xc - ref).max() <= TOL, (lam, "columns")


def test_all_lengths_in_one_ragged_batch():
    lengths = LENGTHS + [0, 1, 0, 1, 5]
    y, off = synth.ragged_chain_batch(lengths, seed0=3)
    w = np.random.default_rng(1).uniform(0, 0.3, size=y.shape).astype(np.float32)
    for weights in (None, w):
        x = _lib.chain_prox(_gpu(y), None if weights is None else _gpu(weights), lam=0.2,
                            offsets=_gpu(off), max_len=max(lengths)).cpu().numpy()
        assert np.abs(x - oracle.chain_solve_batch(y, off, w=weights, lam=0.2)).max() <= TOL


@pytest.mark.parametrize("lam", [0.0, 1e-38, 1e-20, 1e-6])
def test_vanishing_weights_return_y(lam):
    y = synth.chain_batch(9, 300, seed0=1)
    x = _lib.chain_prox(_gpu(y), lam=lam).cpu().numpy()
    assert np.abs(x - y).max() <= 2 * lam + 1e-7


def test_weights_far_above_the_values_take_the_fallback():
    """A cut at a flow above 16 max|y| sends the chain to the warp's dynamic program, alone
    among its neighbours, in rows and columns and for chains of several warps."""
    for n in (400, 1300, 2600):
        y = synth.chain_batch(9, n, seed0=2)
        y[1::3] = (-np.arange(n) / n).astype(np.float32)
        lam = np.float32(n / 16.0)
        w = np.full(y.shape, 0.1, np.float32)
        w[1::3] = lam
        ref = oracle.chain_solve_batch(y.ravel(), np.arange(10) * n, w=w.ravel()).reshape(y.shape)
        x = _lib.chain_prox(_gpu(y), _gpu(w)).cpu().numpy()
        # the values' scale is the weight's: FP32 breakpoints sit near y +- w
        assert np.abs(x - ref).max() <= TOL * max(1.0, lam / 16)
        xc = _lib.chain_prox_columns(_gpu(y.T), _gpu(w.T)).cpu().numpy().T
        assert np.abs(xc - ref).max() <= TOL * max(1.0, lam / 16)


def test_columns_of_a_wider_array():
    H, W, ld = 301, 37, 50
    rng = np.random.default_rng(4)
    y = rng.uniform(0, 1, size=(H, ld)).astype(np.float32)
    yg, x = _gpu(y), torch.full((H, ld), float("nan"), device=DEV)
    lib = _lib.load()
    ws = _lib.workspace(lib.tv_columns_workspace_size(H, W), DEV, "cols")
    _lib._check(lib.tv_chain_solve_columns(_lib._ptr(yg), None, 0.15, H, W, ld, _lib._ptr(x),
                                           _lib._ptr(ws), ws.numel(), _lib._stream(yg.device)))
    g = x.cpu().numpy()
    ref = oracle.chain_solve_batch(np.ascontiguousarray(y[:, :W].T).ravel(), np.arange(W + 1) * H,
                                   lam=0.15).reshape(W, H).T
    assert np.abs(g[:, :W] - ref).max() <= TOL
    assert np.isnan(g[:, W:]).all()

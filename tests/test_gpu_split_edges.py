"""Places where the splitting kernel joins what its lanes, warps and launches hold: runs over lane
and warp boundaries are bitwise equal (the backward pass reads segments off x), images with one
side beyond its longest chain, and phases whose chains take the fallback."""
import numpy as np
import pytest
import torch

import oracle
from paper_1502_07770_gb300 import _lib, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 2e-5


def _gpu(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _solve(y, w, lam):
    x = _lib.chain_prox(_gpu(y), _gpu(w), lam=lam).cpu().numpy()
    xc = _lib.chain_prox_columns(_gpu(y.T), None if w is None else _gpu(w.T), lam=lam).cpu().numpy().T
    return x, xc


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("n", [33, 129, 256, 257, 512, 1024, 1025, 1500, 2048, 2049, 3000, 4095, 4096])
def test_runs_are_bitwise_equal(n, edges):
    rng = np.random.default_rng(n)
    B = 6
    whole = rng.uniform(0, 1, (B, n)).astype(np.float32)                  # one run per chain
    const = np.repeat(rng.uniform(-1, 1, (B, 1)), n, axis=1).astype(np.float32)
    length = rng.integers(20, 600)
    steps = np.repeat(rng.uniform(0, 1, (B, -(-n // length))), length, axis=1)[:, :n].astype(np.float32)
    noisy = (steps + 0.02 * rng.normal(size=steps.shape)).astype(np.float32)
    for name, y, lam in (("whole", whole, 2.0 * n), ("const", const, 0.3), ("steps", steps, 0.05),
                         ("noisy", noisy, 1.0)):
        w = np.full(y.shape, lam, np.float32) * rng.uniform(0.9, 1.1, y.shape).astype(np.float32) if edges else None
        ref = oracle.chain_solve_batch(y.ravel(), np.arange(B + 1) * n, w=None if w is None else w.ravel(),
                                       lam=float(np.float32(lam))).reshape(y.shape)
        fused = np.abs(np.diff(ref, axis=1)) < 1e-12
        if name in ("whole", "const"):
            assert fused.all()
        for x in _solve(y, w, lam):
            assert not (fused & (np.diff(x, axis=1) != 0)).any(), name


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("shape", [(300, 4500), (4500, 300), (70, 4097), (4097, 70), (16, 3000), (12, 4500)])
def test_images_with_one_direction_on_the_splitting_kernel(shape, edges):
    """Rows or columns beyond 4096 nodes, or too many short columns, on the warp- or
    thread-per-chain phases and the other direction on the splitting kernel, the step counter
    advanced by the gap pass and the row phase; both on the old phases (12 x 4500)."""
    f = synth.shapes_image(*shape, seed=sum(shape), n_shapes=60)[1]
    wh, wv = synth.edge_aware_weights(f, 0.2) if edges else (None, None)
    for iters, tol in ((60, 1e-4), (7, 0.0)):
        x, it, gap, ok = _lib.tv2d_denoise(_gpu(f), lam=0.12, w_h=_gpu(wh), w_v=_gpu(wv), max_iters=iters, tol=tol)
        xo, ito, tro, oko = oracle.tv2d_pd(f, lam=0.12, w_h=wh, w_v=wv, max_iters=iters, tol=tol)
        assert it == ito and ok == oko
        assert np.abs(x.cpu().numpy() - xo).max() <= TOL
        assert abs(gap - tro[-1]) <= 1e-6 + 1e-3 * abs(tro[-1])


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("shape", [(400, 400), (404, 1300), (1300, 404)])
def test_phases_with_weights_far_above_the_values(shape, edges):
    """Quadrants of 0, 1/2 and 1 under weights of 30: the halves of a row differ by flows of up
    to side / 8, so rows and columns are cut at flows above 16 max |c| and take the fallback, in
    the initial rows, the dual and the primal phases. Each of the 15 chain solves of 7 iterations
    is off by up to 8 ulp of the weights' size (1.9e-6): 2.4e-4."""
    H, W = shape
    f = (0.5 * (np.arange(H)[:, None] >= H // 2) + 0.5 * (np.arange(W)[None] >= W // 2)).astype(np.float32)
    f += 0.01 * np.random.default_rng(H).normal(size=f.shape).astype(np.float32)
    wh = wv = None
    if edges:  # heavy on every third row and column only
        wh = np.where(np.arange(H)[:, None] % 3 == 0, 30.0, 0.1) * np.ones((H, W - 1))
        wv = np.where(np.arange(W)[None] % 3 == 0, 30.0, 0.1) * np.ones((H - 1, W))
        wh, wv = wh.astype(np.float32), wv.astype(np.float32)
    kw = dict(lam=30.0, w_h=_gpu(wh), w_v=_gpu(wv))
    xo, ito, tro, _ = oracle.tv2d_pd(f, lam=30.0, w_h=wh, w_v=wv, max_iters=7, tol=0.0)
    x, it, gap, _ = _lib.tv2d_denoise(_gpu(f), max_iters=7, tol=0.0, **kw)
    assert it == ito == 7
    assert np.abs(x.cpu().numpy() - xo).max() <= 2.4e-4
    other = synth.shapes_image(60, 80, seed=1, n_shapes=9)[1]  # a plain image beside it
    xs, its, gaps, _ = _lib.tv2d_denoise_batched([_gpu(f), _gpu(other)], [30.0, 0.1], [_gpu(wh), None],
                                                 [_gpu(wv), None], max_iters=7, tol=0.0)
    assert np.abs(xs[0].cpu().numpy() - xo).max() <= 2.4e-4
    xp = oracle.tv2d_pd(other, lam=0.1, max_iters=7, tol=0.0)[0]
    assert np.abs(xs[1].cpu().numpy() - xp).max() <= TOL

"""The 2D phases on the threshold-splitting kernel where a side takes two or four warps a chain,
with the gap pass inside the column phase's launch (batches of 6, then 3 iterations), single
images and batches, against the oracle; and the non-convex chains around the sizes of their
striped lists. Tolerances are those of the drivers' own parity tests."""
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


def _image(h, w, seed):
    return synth.shapes_image(h, w, seed=seed, n_shapes=max(2, h * w // 400))[1]


SHAPES = [(31, 33), (32, 64), (65, 31), (12, 1100), (1100, 12), (1030, 33), (5, 2100), (2100, 5)]


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_single_images(shape, edges):
    f = _image(*shape, seed=sum(shape))
    wh, wv = synth.edge_aware_weights(f, 0.2) if edges else (None, None)
    for iters, tol in ((60, 1e-4), (7, 0.0), (10, 0.0)):
        x, it, gap, ok = _lib.tv2d_denoise(_gpu(f), lam=0.12, w_h=_gpu(wh), w_v=_gpu(wv),
                                           max_iters=iters, tol=tol)
        xo, ito, tro, oko = oracle.tv2d_pd(f, lam=0.12, w_h=wh, w_v=wv, max_iters=iters, tol=tol)
        assert it == ito and ok == oko
        assert np.abs(x.cpu().numpy() - xo).max() <= TOL
        assert abs(gap - tro[-1]) <= 1e-6 + 1e-3 * abs(tro[-1])


@pytest.mark.parametrize("edges", [False, True])
def test_batched_images(edges):
    fs = [_image(*s, seed=7 + sum(s)) for s in SHAPES]
    lams = [0.05 + 0.03 * m for m in range(len(fs))]
    ws = [synth.edge_aware_weights(f, lam) if edges and m % 3 else (None, None)
          for m, (f, lam) in enumerate(zip(fs, lams))]
    y0s = [None] * len(fs)
    for m in (2, 4):  # a warm start, also where a side takes two warps
        y0s[m] = (0.02 * _image(*SHAPES[m], seed=90 + m)).astype(np.float32)
    xs, its, gaps, ok = _lib.tv2d_denoise_batched(
        [_gpu(f) for f in fs], lams, [_gpu(w[0]) for w in ws], [_gpu(w[1]) for w in ws],
        [_gpu(y) for y in y0s], max_iters=100, tol=1e-4)
    assert ok
    for m, f in enumerate(fs):
        xo, ito, tro, _ = oracle.tv2d_pd(f, lam=lams[m], w_h=ws[m][0], w_v=ws[m][1], y0=y0s[m],
                                         max_iters=100, tol=1e-4)
        assert its[m] == ito, m
        assert np.abs(xs[m].cpu().numpy() - xo).max() <= TOL, m
        assert abs(gaps[m] - tro[-1]) <= 1e-6 + 1e-3 * abs(tro[-1]), m


@pytest.mark.parametrize("C", [float("inf"), 0.7])
@pytest.mark.parametrize("labels", [1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 256, 257, 300])
def test_nonconvex_list_sizes(labels, C):
    """Breakpoints 0 .. labels - 1 of every node (all duplicates in the merges): lists of just
    under, at and over 32 points a stripe, and unaries beyond what is fetched ahead."""
    rng = np.random.default_rng(labels)
    R, n = 3, 9
    cost = rng.uniform(0.0, 2.0, (R, n, labels)).astype(np.float32)
    x, e = _lib.chain_prox_nonconvex(_gpu(cost), sl=-1.5, sr=0.75, w=0.25, C=C, max_breakpoints=1024)
    st, _ = _lib.workspace_status(_lib.workspace(1, DEV, "nonconvex"))
    assert st == _lib.TV_OK
    lab = np.arange(labels, dtype=np.float64)
    x, e = x.cpu().numpy().reshape(R, n), e.cpu().numpy()
    us = [(lab, cost[r, i].astype(np.float64), -1.5, 0.75) for r in range(R) for i in range(n)]
    w, c = np.full(R * n, 0.25), np.full(R * n, C)
    _, eo = oracle.chain_solve_nonconvex(us, w, c, np.arange(R + 1) * n)
    for r in range(R):
        assert abs(e[r] - eo[r]) <= 1e-4 + 1e-5 * abs(eo[r])
        z = x[r].astype(np.float64)  # x reaches the energy
        ex = sum(np.interp(v, lab, cost[r, i]) + (-1.5 * min(v, 0.0) if v < 0 else 0.75 * max(v - lab[-1], 0.0))
                 for i, v in enumerate(z)) + np.minimum(0.25 * np.abs(np.diff(z)), C).sum()
        assert abs(ex - eo[r]) <= 1e-4 + 1e-5 * abs(eo[r])

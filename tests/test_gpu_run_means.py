"""The backward kernel of chains that fit a warp's registers (csrc/tv_grad.cu,
run_means_kernel) against float64 segment means.

Gradients are N(0, 1): a mean of k of them, summed in FP32, is off by at most k / 2 + 2 ulp of
the largest partial sum over k, below 2e-6 for the runs here (up to 4096 nodes, partial sums
below 300).
"""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 2e-6


def _solution(n, rng):
    """A piecewise-constant row: single nodes, short runs, and runs longer than a lane."""
    out, top = [], int(rng.choice([2, 12, 100, 5000]))
    while sum(map(len, out)) < n:
        out.append(np.full(int(rng.integers(1, top + 1)), rng.normal()))
    return np.concatenate(out)[:n].astype(np.float32)


def _reference(x, g):
    cut = np.flatnonzero(np.r_[True, x[1:] != x[:-1]])
    cnt = np.diff(np.r_[cut, len(x)])
    m = np.repeat(np.add.reduceat(g.astype(np.float64), cut) / cnt, cnt)
    gw = np.zeros(len(x))
    gw[:-1] = np.sign(x[1:] - x[:-1]) * (m[:-1] - m[1:])
    return m, gw


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 31, 32, 33, 255, 256, 257, 512, 513, 768, 769, 1023,
                               1024, 1025, 1536, 1537, 2048, 2049, 3073, 4095, 4096])
def test_rows(n):
    rng = np.random.default_rng(n)
    x = np.stack([_solution(n, rng) for _ in range(7)])
    g = rng.normal(size=x.shape).astype(np.float32)
    ref = [_reference(a, b) for a, b in zip(x, g)]
    for shift in (0, 1):  # 16-byte accesses, and arrays off the 16-byte grid
        xs, gs = (torch.empty(x.size + shift, device=DEV)[shift:].view(x.shape) for _ in range(2))
        xs.copy_(_gpu(x))
        gs.copy_(_gpu(g))
        gy, gw = _lib.chain_prox_backward(xs, gs, with_w=True)
        assert np.abs(gy.cpu().numpy() - np.stack([r[0] for r in ref])).max() <= TOL
        assert np.abs(gw.cpu().numpy() - np.stack([r[1] for r in ref])).max() <= 2 * TOL
        assert torch.equal(_lib.chain_prox_backward(xs, gs)[0], gy)


def test_csr_classes_and_unwritten_entries():
    """One batch over every length class; nothing outside the chains is written, nor (by
    tv_chain_solve_backward) grad_w at a chain's last node."""
    rng = np.random.default_rng(0)
    lengths = [0, 1, 700, 2, 1024, 1025, 0, 2048, 2049, 33, 4096, 5]
    off = np.r_[0, np.cumsum(lengths)] + 3
    total = int(off[-1]) + 5
    x = np.zeros(total, np.float32)
    for k, n in enumerate(lengths):
        x[off[k]:off[k + 1]] = _solution(n, rng) if n else []
    g = rng.normal(size=total).astype(np.float32)
    xg, gg, og = _gpu(x), _gpu(g), _gpu(off.astype(np.int64))
    gy, gw = (torch.full((total,), float("nan"), device=DEV) for _ in range(2))
    ws = _lib.workspace(256, DEV, "grad-csr")
    lib = _lib.load()
    _lib._check(lib.tv_chain_solve_backward(_lib._ptr(xg), _lib._ptr(gg), _lib._ptr(og),
                                            len(lengths), max(lengths), _lib._ptr(gy),
                                            _lib._ptr(gw), _lib._ptr(ws), ws.numel(),
                                            _lib._stream(torch.device(DEV))))
    assert _lib.workspace_status(ws)[0] == _lib.TV_OK
    gy, gw = gy.cpu().numpy(), gw.cpu().numpy()
    seen = np.zeros(total, bool)
    for k, n in enumerate(lengths):
        if not n:
            continue
        a, b = off[k], off[k + 1]
        m, w = _reference(x[a:b], g[a:b])
        assert np.abs(gy[a:b] - m).max() <= TOL
        assert n == 1 or np.abs(gw[a:b - 1] - w[:-1]).max() <= 2 * TOL
        assert np.isnan(gw[b - 1])
        seen[a:b] = True
    assert np.isnan(gy[~seen]).all() and np.isnan(gw[~seen]).all()


def test_nonfinite_gradients_stay_in_their_run():
    rng = np.random.default_rng(1)
    n = 1500
    x = np.repeat(rng.normal(size=n // 5), 5).astype(np.float32)[None]
    g = rng.normal(size=(1, n)).astype(np.float32)
    g[0, 52], g[0, 1001] = np.inf, np.nan
    gy = _lib.chain_prox_backward(_gpu(x), _gpu(g))[0].cpu().numpy()[0]
    bad = np.zeros(n, bool)
    bad[50:55] = bad[1000:1005] = True
    assert not np.isfinite(gy[bad]).any() and np.isfinite(gy[~bad]).all()

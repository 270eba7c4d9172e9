"""Which backward kernel a batch takes: the register kernel has a launch per class of lengths (up
to 1024, 2048 and 4096 nodes) for CSR batches, the step-wise one a launch for all, and takes
large batches of short chains. Results on both sides of each line against float64 means (sums of
up to 2500 gradients N(0, 1) in FP32: 1e-5)."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _problem(off, seed):
    rng = np.random.default_rng(seed)
    n = int(off[-1])
    x = np.repeat(rng.normal(size=n), rng.integers(1, 9, n))[:n].astype(np.float32)
    g = rng.normal(size=n).astype(np.float32)
    head = np.r_[True, x[1:] != x[:-1]]
    head[off[:-1]] = True  # (no empty chains)
    cut = np.flatnonzero(head)
    cnt = np.diff(np.r_[cut, n])
    m = np.add.reduceat(g.astype(np.float64), cut) / cnt
    m = np.repeat(m, cnt)
    gw = np.zeros(n)
    gw[:-1] = np.where(head[1:], np.sign(x[1:] - x[:-1]) * (m[:-1] - m[1:]), 0.0)
    gw[off[1:] - 1] = 0.0
    return x, g, m, gw


def _check(x, g, m, gw, launches, **kw):
    xg, gg = (torch.from_numpy(a).to(DEV) for a in (x, g))
    n0 = _lib.load().tv_launch_count()
    gy, gwg = _lib.chain_prox_backward(xg, gg, with_w=True, **kw)
    assert _lib.load().tv_launch_count() - n0 == launches
    assert np.abs(gy.cpu().numpy().ravel() - m).max() <= 1e-5
    assert np.abs(gwg.cpu().numpy().ravel() - gw).max() <= 2e-5


@pytest.mark.parametrize("chains,longest,launches", [
    (2000, 2500, 3), (24000, 2500, 3), (24001, 2500, 1), (200000, 2500, 1), (4096, 1500, 2), (4097, 1500, 1),
    (2048, 700, 1), (2049, 700, 1), (100000, 700, 1)])
def test_csr(chains, longest, launches):
    r = np.random.default_rng(chains).integers(1, 40, chains)
    r[chains // 3] = longest
    off = np.r_[0, np.cumsum(r)]
    _check(*_problem(off, chains), launches, offsets=torch.from_numpy(off).to(DEV), max_len=longest)


@pytest.mark.parametrize("n", [1, 20, 127, 128])
@pytest.mark.parametrize("chains", [4096, 4097])
def test_rows(n, chains):
    x, g, m, gw = _problem(np.arange(chains + 1) * n, n)
    _check(x.reshape(chains, n), g.reshape(chains, n), m, gw, 1)

"""Which kernel a CSR batch takes, told by its launches: the splitting kernel has one per class
of lengths (up to 1024, 2048 and 4096 nodes), the thread kernels one for all. Batches for which
it was measured faster stay on the splitting kernel; large ones, whose chains are mostly far
shorter than the longest or too many for warps of their own, go to the thread kernels. Results
against the oracle either way."""
import numpy as np
import pytest
import torch

import oracle
from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lengths(kind, chains, longest):
    r = np.random.default_rng(chains + longest).integers(1, (longest if kind == "even" else 40) + 1, chains)
    r[chains // 2] = longest
    return r


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("kind,chains,longest,split", [
    ("one", 200000, 1100, False), ("one", 50000, 1100, False), ("one", 5000, 1100, True), ("one", 9000, 4096, True),
    ("even", 40000, 1100, False), ("even", 6000, 2500, True), ("even", 3000, 4000, True)])
def test_route(kind, chains, longest, split, edges):
    r = _lengths(kind, chains, longest)
    off = np.r_[0, np.cumsum(r)]
    rng = np.random.default_rng(1)
    y = (np.repeat(rng.uniform(0, 1, off[-1] // 12 + 1), 12)[:off[-1]] + 0.1 * rng.normal(size=off[-1])).astype(np.float32)
    w = rng.uniform(0, 0.3, y.size).astype(np.float32) if edges else None
    g = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    yg, wg, og = g(y), g(w), g(off)
    n0 = _lib.load().tv_launch_count()
    x = _lib.chain_prox(yg, wg, lam=0.2, offsets=og, max_len=longest)
    launches = _lib.load().tv_launch_count() - n0
    assert launches == (1 if not split else 2 if longest <= 2048 else 3)
    x = x.cpu().numpy()
    for k in (0, chains // 2, chains // 2 + 1, chains - 1):
        s = slice(off[k], off[k + 1])
        ref = oracle.chain_solve_batch(y[s], np.array([0, r[k]]), w=None if w is None else w[s], lam=0.2)
        assert np.abs(x[s] - ref).max() <= 2e-5

"""The autotuner and the library's own limits: they go with length, layout and weights, and one
crossover for every batch replaces them only where it is faster (no GPU); what autotune() applies
on this GPU leaves every batch on its kernel (the bits of the results tell)."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib, autotune


def test_choice():
    assert autotune.keep_limits([1.0, 2.0], [1.0, 2.0])
    assert autotune.keep_limits([1.0, 1.0], [0.99, 1.0])     # within the margin
    assert autotune.keep_limits([1.0, 1.0], [0.9, 2.0])
    assert not autotune.keep_limits([1.0, 1.0], [0.9, 0.9])


def test_what_is_applied(monkeypatch):
    applied = []
    monkeypatch.setattr(_lib, "set_coop_max_chains", applied.append)
    monkeypatch.setattr(_lib, "set_batched_warps", lambda v: None)
    autotune.apply({"coop_max_chains": 4096, "batched_warps": 4, "keep_limits": True})
    autotune.apply({"coop_max_chains": 4096, "batched_warps": 4, "keep_limits": False})
    autotune.apply({"coop_max_chains": 2048, "batched_warps": 4})
    assert applied == [0, 4096, 2048]


def test_caches_of_the_old_limits_lapse():
    assert _lib.load().tv_version() > 100


@pytest.mark.gpu
def test_batches_stay_on_their_kernels(tmp_path):
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(3)
    rand = lambda *s: torch.rand(s, generator=g, device=dev)
    off = torch.from_numpy(np.r_[0, np.cumsum(np.random.default_rng(0).integers(1, 2501, 6000))]).to(dev)
    y, w = rand(int(off[-1])), 0.2 * rand(int(off[-1]))
    yr, wr, yc, yt = rand(8000, 385), 0.2 * rand(8000, 385), rand(512, 9000), rand(9000, 1024)
    calls = [lambda: _lib.chain_prox(y, w=w, offsets=off, max_len=2500), lambda: _lib.chain_prox(yr, w=wr),
             lambda: _lib.chain_prox_columns(yc, lam=0.1), lambda: _lib.chain_prox(yt, lam=0.1)]
    before = [c() for c in calls]
    try:
        params = autotune.autotune(path=str(tmp_path / "tune.json"))
        after = [c() for c in calls]
    finally:
        _lib.set_coop_max_chains(0)
        _lib.set_batched_warps(4)
    assert params["keep_limits"], params["mixed_ms"]
    for a, b in zip(before, after):
        assert torch.equal(a, b)

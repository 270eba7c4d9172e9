"""Which kernel a uniform batch of tv_chain_solve or tv_chain_solve_columns takes by default, told
by the bits of its result: the splitting kernel and the thread kernels round differently. The
cases lie on both sides of lines where the one or the other was measured faster."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("cols,n,chains,edges,split", [
    (False, 1027, 7000, False, True), (False, 1027, 20000, False, False),
    (False, 2050, 7000, False, True), (False, 2050, 9000, False, False), (False, 3001, 9000, False, True),
    (False, 300, 6500, False, True), (False, 300, 8192, False, False), (False, 512, 8192, False, True),
    (False, 385, 7000, False, True), (False, 385, 8192, False, False),
    (False, 201, 30000, True, True), (False, 201, 50000, True, False), (False, 385, 50000, True, True),
    (True, 300, 40000, False, True), (True, 300, 100000, False, False), (True, 512, 100000, False, True)])
def test_route(cols, n, chains, edges, split):
    g = torch.Generator(device=DEV).manual_seed(n + chains)
    shape = (n, chains) if cols else (chains, n)
    y = torch.rand(shape, generator=g, device=DEV)
    w = 0.1 * torch.rand(shape, generator=g, device=DEV) if edges else None
    solve = _lib.chain_prox_columns if cols else _lib.chain_prox
    default = solve(y, w, lam=0.07)
    forced = {}
    try:
        for name, most in (("split", 1 << 40), ("thread", 1)):
            _lib.set_coop_max_chains(most)
            forced[name] = solve(y, w, lam=0.07)
    finally:
        _lib.set_coop_max_chains(0)
    assert not torch.equal(forced["split"], forced["thread"])
    assert torch.equal(default, forced["split" if split else "thread"])


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("cols,n,split", [(False, 8, False), (False, 19, False), (False, 20, True), (False, 40, True),
                                          (True, 8, False), (True, 31, False), (True, 32, True), (True, 48, True)])
def test_short_chains(cols, n, split, edges):
    """Short chains stay on the warp's dynamic program (below 64 nodes solve mode 0 is the
    default's), which is the faster one for them."""
    chains = 3000
    g = torch.Generator(device=DEV).manual_seed(n)
    shape = (n, chains) if cols else (chains, n)
    y = torch.rand(shape, generator=g, device=DEV)
    w = 0.1 * torch.rand(shape, generator=g, device=DEV) if edges else None
    solve = _lib.chain_prox_columns if cols else _lib.chain_prox
    default = solve(y, w, lam=0.07)
    try:
        _lib.set_coop_max_chains(1 << 40)
        splitting = solve(y, w, lam=0.07)
        _lib.set_coop_split(0)
        program = solve(y, w, lam=0.07)
    finally:
        _lib.set_coop_max_chains(0)
        _lib.set_coop_split(1)
    assert not torch.equal(splitting, program)
    assert torch.equal(default, splitting if split else program)

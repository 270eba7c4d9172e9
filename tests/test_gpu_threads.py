"""Calls from several host threads at once, each with a stream, arrays and a workspace of its own.

A kernel's shared-memory limit belongs to the process: a call may not lower it between another
call's opt-in and its launch. The pairs of calls run the same kernel with blocks of two sizes."""
import threading

import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CALLS, BATCH = 6000, 64


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device=DEV)


def _columns(H, W=8):
    """tv_chain_solve_columns as (call(stream), result)."""
    lib = _lib.load()
    y = torch.from_numpy(np.ascontiguousarray(synth.chain_batch(W, H, seed0=H).T)).to(DEV)
    x, ws = torch.empty_like(y), _bytes(lib.tv_columns_workspace_size(H, W))
    args = (_lib._ptr(y), None, 0.2, H, W, W, _lib._ptr(x), _lib._ptr(ws), ws.numel())
    return lambda s: lib.tv_chain_solve_columns(*args, s), x, (y, ws)


def _backward(n, B=8):
    lib = _lib.load()
    x = torch.from_numpy(synth.chain_batch(B, n, seed0=n).round(1)).to(DEV)
    g = torch.from_numpy(synth.chain_batch(B, n, seed0=n + 1)).to(DEV)
    gy, ws = torch.empty_like(x), _bytes(256)
    args = (_lib._ptr(x), _lib._ptr(g), None, B, n, _lib._ptr(gy), None, _lib._ptr(ws), 256)
    return lambda s: lib.tv_chain_solve_backward(*args, s), gy, (x, g, ws)


def _nonconvex(labels):
    lib = _lib.load()
    cost = torch.from_numpy(np.random.default_rng(labels).uniform(0, 2, (2, 5, labels)).astype(np.float32)).to(DEV)
    T = 4 * labels
    x, e = torch.empty(10, device=DEV), torch.empty(2, dtype=torch.float64, device=DEV)
    ws = _bytes(lib.tv_chain_nonconvex_workspace_size(10, 2, 5, T))
    args = (None, None, _lib._ptr(cost), labels, None, None, -1.0, 1.0, None, 0.25, None, 0.7, None, 10, 2, 5, T,
            _lib._ptr(x), _lib._ptr(e), _lib._ptr(ws), ws.numel())
    return lambda s: lib.tv_chain_solve_nonconvex(*args, s), x, (cost, e, ws)


PAIRS = {"columns": lambda: (_columns(4096), _columns(3073)),
         "backward": lambda: (_backward(4096), _backward(2100)),
         "nonconvex": lambda: (_nonconvex(250), _nonconvex(8))}


@pytest.mark.parametrize("pair", PAIRS)
def test_two_threads(pair):
    jobs = PAIRS[pair]()
    want = []
    for call, out, _ in jobs:
        assert call(_lib._stream(torch.device(DEV))) == _lib.TV_OK
        torch.cuda.synchronize()
        want.append(out.clone())
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    failed = []

    def work(call, stream):
        s = _lib.ctypes.c_void_p(stream.cuda_stream)
        for k in range(CALLS):
            if call(s) != _lib.TV_OK:
                failed.append((k, _lib.load().tv_last_error()))
                return
            if k % BATCH == BATCH - 1:
                stream.synchronize()

    threads = [threading.Thread(target=work, args=(job[0], s)) for job, s in zip(jobs, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for job, ref in zip(jobs, want):
        assert torch.equal(job[1], ref)

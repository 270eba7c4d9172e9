"""A batch whose initial duals lie in memory that the solve writes: the results are those of
copies of the duals, bit for bit, in one iteration and in many, and with the dual asked for."""
import numpy as np
import pytest
import torch

from paper_1502_07770_gb300 import _lib, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("iters", [0, 1, 7])
def test_duals_in_the_outputs(iters):
    H, W = 45, 70
    n = H * W
    fs = [torch.from_numpy(synth.shapes_image(H, W, seed=m, n_shapes=20)[1]).to(DEV) for m in range(4)]
    duals = [torch.from_numpy((0.03 * synth.shapes_image(H, W, seed=50 + m, n_shapes=20)[1]).astype(np.float32)).to(DEV)
             for m in range(4)]
    lams = [0.1, 0.15, 0.2, 0.12]
    apart = [torch.empty_like(d) for d in duals]
    ref, rit, _, _ = _lib.tv2d_denoise_batched(fs, lams, y0s=[d.clone() for d in duals], max_iters=iters, tol=0.0,
                                               y_outs=apart)
    # image 0 starts from image 1's output, 1 from 13 floats before its own, 2 from 5 after image
    # 0's and into 3's, 3 from a buffer of its own that also takes its final dual
    buf = torch.zeros(6 * n, device=DEV)
    at = lambda o: buf[o:o + n].view(H, W)
    xs = [at(0), at(2 * n), at(4 * n), at(n)]
    y0s = [xs[1], at(2 * n - 13), at(5), duals[3].clone()]
    y_outs = [torch.empty_like(d) for d in duals[:3]] + [y0s[3]]
    for order in ((0,), (1,), (2,)):  # (they overlap each other: one of them at a time)
        start = [duals[m].clone() for m in range(3)] + [y0s[3]]
        for m in order:
            start[m] = y0s[m]
        for m in range(4):
            start[m].copy_(duals[m])
        out, it, _, _ = _lib.tv2d_denoise_batched(fs, lams, y0s=start, max_iters=iters, tol=0.0, outs=xs,
                                                  y_outs=y_outs)
        assert it == rit
        for m in range(4):
            assert torch.equal(out[m], ref[m]), (order, m)
            assert torch.equal(y_outs[m], apart[m]), (order, m)

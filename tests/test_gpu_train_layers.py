"""The training step's kernels (grouped layout on tcgen05, ReLU masks as bits, one-channel
head and first layer) against the general NHWC kernels composed to the same gradient, at the
edges of the 8 x 16 and 128-pixel tiles and of the head's 16-row strips."""
import pytest
import torch

from paper_1502_07770_gb300 import _lib, learned

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _general(net, f, lam, target):
    """Loss and gradient through pack_input, conv3x3, dual_head and the NHWC backward kernels."""
    lib, s, vp = net.lib, _lib._stream(net.device), learned._vp
    B, H, W = f.shape
    n, bf = B * H * W, torch.bfloat16
    ws = torch.empty(lib.tv_net_workspace_size(B, H, W), dtype=torch.uint8, device=DEV)
    x = torch.empty(n * 16, dtype=bf, device=DEV)
    _lib._check(lib.tv_net_pack_input(vp(f), B, H, W, vp(lam), vp(x), s))
    xs, pres = [x], []
    for (cin, cout, relu), (w, b) in zip(learned.LAYERS, net.offsets):
        pre = torch.empty(n * cout, device=DEV)
        act = torch.empty(n * cout, dtype=bf, device=DEV)
        _lib._check(lib.tv_net_conv3x3(vp(xs[-1]), B, H, W, cin, vp(net.params_bf16, w), vp(net.params, b),
                                       cout, int(relu), vp(pre), vp(act), s))
        xs.append(act)
        pres.append(pre)
    y, loss = torch.empty(n, device=DEV), torch.empty(1, device=DEV)
    dy = torch.empty(n * 16, dtype=bf, device=DEV)
    _lib._check(lib.tv_net_dual_head(vp(pres[-1]), B, H, W, vp(lam), vp(target), vp(y), vp(loss), vp(dy),
                                     vp(ws), ws.numel(), s))
    grad = torch.zeros_like(net.grad)
    flip = torch.empty(32 * 9 * 32, dtype=bf, device=DEV)
    for li in range(len(learned.LAYERS) - 1, -1, -1):
        (cin, cout, _), (w, b) = learned.LAYERS[li], net.offsets[li]
        _lib._check(lib.tv_net_conv3x3_backward_weight(vp(xs[li]), vp(dy), B, H, W, cin, cout,
                                                       vp(grad, w), vp(grad, b), vp(ws), ws.numel(), s))
        if li:
            dx = torch.empty(n * cin, dtype=bf, device=DEV)
            _lib._check(lib.tv_net_conv3x3_backward_data(vp(dy), B, H, W, cout, vp(net.params_bf16, w), cin,
                                                         vp(pres[li - 1]), vp(dx), vp(flip), s))
            dy = dx
    return loss, grad


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 2, 15), (2, 8, 16), (1, 9, 17), (3, 16, 127), (2, 17, 128),
                                   (1, 33, 129), (70, 7, 5), (1, 300, 260)])
def test_training_kernels_match_the_general_ones(shape):
    """Both sides round to BF16 at the same places and add the same products in FP32, in
    another order: per block at most a few thousand of them, so about 1e-5 of a layer's
    gradient; a BF16 rounding that such a difference flips moves one of the summed products by
    2^-8, which 1e-3 of the norm leaves room for, while a misplaced or missing pixel does not
    fit in it."""
    net = learned.WarmStartNet(DEV, seed=4)
    net.params[net.offsets[-1][0]:net.offsets[-1][1]] *= 10.0
    net._refresh_bf16()
    g = torch.Generator().manual_seed(sum(shape))
    f = torch.rand(shape, generator=g).to(DEV)
    lam = (0.05 + 0.25 * torch.rand(shape[0], generator=g)).to(DEV)
    target = (torch.randn(shape, generator=g) * 0.05).to(DEV)
    t0 = net.lib.tv_net_tensor_timeouts()
    loss = net.loss_and_grad(f, lam, target)
    assert net.lib.tv_net_tensor_timeouts() == t0
    wloss, want = _general(net, f, lam, target)
    assert abs(loss.item() - wloss.item()) <= 1e-5 * abs(wloss.item())
    for (cin, cout, _), (w, b) in zip(learned.LAYERS, net.offsets):
        for a, n in ((w, cout * 9 * cin), (b, cout)):
            got, ref = net.grad[a:a + n].double(), want[a:a + n].double()
            assert (got - ref).norm() <= 1e-3 * ref.norm()

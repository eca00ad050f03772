"""The marching weight gradient with repeated drains (GB300): volumes over the rule that
keeps shorter sums on the row-splitting kernel, every CTA with several columns' planes
and more products than its accumulators take between drains."""
import numpy as np
import pytest

from oracle import wsnet_oracle as N
from test_gpu_wsnet import _bf16, _he, _padded, torch  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPE = (5, 500, 8, 14)  # B, Z, Y, X: planes of 128 rows, 8 products each


def _rule(torch, shape, splits, sets):  # noqa: F811
    """Products of 16 interior rows that an accumulator may take, and that a CTA has in
    all (`sets` CTAs share a plane)."""
    B, Z, Y, X = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    limit = 17 * B * Z * Y * (X + 2) // (16 * splits * sms * 16)
    return limit, B * Z * (Y * (X + 2) // 16) // (sms // sets)


@pytest.mark.parametrize("cin,cout,splits,sets", [(32, 32, 2, 1), (32, 64, 2, 3), (64, 32, 2, 2), (64, 64, 1, 3)])
def test_weight_gradient_with_drains(torch, cin, cout, splits, sets):  # noqa: F811
    """Onto a preset buffer, against the FP64 oracle; bound of test_gpu_march.py."""
    from paper_1806_10589_gb300 import conv3d_bf16

    B, Z, Y, X = SHAPE
    limit, products = _rule(torch, SHAPE, splits, sets)
    assert 63 <= limit < products, (limit, products)
    rng = np.random.default_rng(cin + 3 * cout)
    ta, a = _padded(torch, rng.standard_normal((B, cin, Z, Y, X)))
    tg, g = _padded(torch, rng.standard_normal((B, cout, Z, Y, X)))
    w = _bf16(torch, np.zeros((cout, 27, cin))).cuda()
    gw = torch.full((cout, 27, cin), 0.5, dtype=torch.float32, device="cuda")
    conv3d_bf16(2, ta.data_ptr(), tg.data_ptr(), w.data_ptr(), 0, 0, gw.data_ptr(), B, X, Y, Z, cin, cout,
                torch.cuda.current_stream())
    ref, S = 0.0, 0.0
    w0 = np.zeros((cout, cin, 27))
    for b in range(B):
        ref = ref + N.conv_backward(a[b], w0, g[b])[1]
        S = S + N.conv_backward(np.abs(a[b]), w0, np.abs(g[b]))[1]
    got = gw.double().cpu().numpy().transpose(0, 2, 1) - 0.5
    assert (np.abs(got - ref) <= 2.0 ** -15 * (S + 0.5)).all()


@pytest.mark.parametrize("base,splits,sets", [(32, 2, 1), (64, 1, 3)])
def test_network_gradient_with_drains(torch, base, splits, sets):  # noqa: F811
    """The same on the network's own partial sums: twice bitwise the same, and against
    the oracle at the bounds of test_loss_and_gradient_match_oracle."""
    from paper_1806_10589_gb300 import WarmStartNet

    B, shape = SHAPE[0], SHAPE[1:]
    limit, products = _rule(torch, SHAPE, splits, sets)
    assert 63 <= limit < products, (limit, products)
    rng = np.random.default_rng(base)
    masks = (rng.random((B,) + shape) < 0.35).astype(np.uint8)
    targets = rng.standard_normal((B, N.NOUT) + shape).astype(np.float32)
    p = _he(1, base, 5)
    net = WarmStartNet(1, base, stream=torch.cuda.current_stream())
    try:
        net.set_params(p)
        loss, g = net.loss_grad(masks, targets)
        _, again = net.loss_grad(masks, targets)
    finally:
        net.close()
    np.testing.assert_array_equal(g, again)
    npore = float((masks == 0).sum())
    ref_loss, ref_g = 0.0, np.zeros(p.size)
    for b in range(B):
        nb = float((masks[b] == 0).sum())
        lb, gb = N.loss_and_grad(p.astype(np.float64), 1.0 - masks[b], targets[b], 1, base)
        ref_loss += lb * nb / npore
        ref_g += gb * nb / npore
    assert abs(loss - ref_loss) <= 1e-2 * ref_loss, (loss, ref_loss)
    k = 0
    for li, (co, ci) in enumerate(N.layer_shapes(1, base)):
        n = co * 27 * ci + co
        rel = np.linalg.norm(g[k:k + n] - ref_g[k:k + n]) / np.linalg.norm(ref_g[k:k + n])
        assert rel <= 0.06, (li, co, ci, rel)
        k += n

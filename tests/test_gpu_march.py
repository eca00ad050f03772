"""The marching convolution and weight-gradient kernels with many planes per CTA
(GB300), against the FP64 oracle.

These kernels give a CTA a run of (sample, patch, plane) items; a volume with fewer
items than SMs gives it one.  Here every CTA gets several: accumulators and plane
buffers are used again (three and up to four of each), a run crosses from one column
to the next inside a CTA, and the weight gradient drains its accumulators more than
once, onto the caller's buffer (single calls) and onto its own partial sums (network).
Forward and data gradient are held to the bounds derived in test_gpu_wsnet.py.  A
weight is a sum of at most 64 truncating additions per accumulator (2^-23 each) and
of at most 200 drained sums (2^-24 each), under 2^9 roundings of 2^-24: 2^-15 of the
sum of absolute values."""
import numpy as np
import pytest

from oracle import wsnet_oracle as N
from test_gpu_wsnet import _bf16, _he, _padded, _unpad, torch  # noqa: F401

pytestmark = pytest.mark.gpu

TALL = (3, 500, 8, 14)   # B, Z, Y, X: one patch of 128 rows a plane
WIDE = (2, 160, 20, 40)  # several patches a plane


@pytest.mark.parametrize("cin,cout,shape", [(32, 32, TALL), (32, 64, TALL), (64, 32, TALL), (64, 64, TALL),
                                            (32, 32, WIDE), (64, 64, WIDE)])
def test_conv_of_many_planes_per_cta(torch, cin, cout, shape):  # noqa: F811
    from paper_1806_10589_gb300 import conv3d_bf16

    B, Z, Y, X = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert B * Z > 2 * sms, "at least three planes in some CTAs, whatever the patch"
    assert B * Z * (Y * (X + 2) // 16) > 64 * sms, "more products per CTA than an accumulator takes"
    rng = np.random.default_rng(cin + 3 * cout + X)
    ta, a = _padded(torch, rng.standard_normal((B, cin, Z, Y, X)))
    tg, g = _padded(torch, rng.standard_normal((B, cout, Z, Y, X)))
    wb = _bf16(torch, rng.standard_normal((cout, 27, cin)) / np.sqrt(27 * cin))
    w = wb.double().numpy().transpose(0, 2, 1)
    tw = wb.cuda().contiguous()
    bias = rng.standard_normal(cout).astype(np.float32)
    tb = torch.tensor(bias).cuda()
    st = torch.cuda.current_stream()
    out = torch.full((B, Z + 2, Y + 2, X + 2, cout), 7.0, dtype=torch.bfloat16, device="cuda")
    gin = torch.full((B, Z + 2, Y + 2, X + 2, cin), 7.0, dtype=torch.bfloat16, device="cuda")
    gw = torch.full((cout, 27, cin), 0.5, dtype=torch.float32, device="cuda")
    conv3d_bf16(0, ta.data_ptr(), 0, tw.data_ptr(), tb.data_ptr(), 1, out.data_ptr(), B, X, Y, Z, cin, cout, st)
    conv3d_bf16(1, tg.data_ptr(), 0, tw.data_ptr(), 0, 0, gin.data_ptr(), B, X, Y, Z, cin, cout, st)
    conv3d_bf16(2, ta.data_ptr(), tg.data_ptr(), tw.data_ptr(), 0, 0, gw.data_ptr(), B, X, Y, Z, cin, cout, st)
    for t in (out, gin):
        border = t.clone()
        border[:, 1:-1, 1:-1, 1:-1, :] = 0
        assert not border.any(), "border rows must be written 0"
    ref_w, S_w = 0.0, 0.0
    for b in range(B):
        b64 = bias.astype(np.float64)
        ref = N.relu(N.conv(a[b], w, b64))
        S = N.conv(np.abs(a[b]), np.abs(w), np.abs(b64))
        assert (np.abs(_unpad(out[b:b + 1])[0] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), "forward"
        ref, rw, _ = N.conv_backward(a[b], w, g[b])
        S, sw, _ = N.conv_backward(np.abs(a[b]), np.abs(w), np.abs(g[b]))
        assert (np.abs(_unpad(gin[b:b + 1])[0] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), "data gradient"
        ref_w, S_w = ref_w + rw, S_w + sw
    got = gw.double().cpu().numpy().transpose(0, 2, 1) - 0.5
    assert (np.abs(got - ref_w) <= 2.0 ** -15 * (S_w + 0.5)).all(), "weight gradient"


def test_network_gradient_of_many_planes_per_cta(torch):  # noqa: F811
    """The same through the network (two levels, all four channel pairs), whose weight
    gradients go through partial sums: twice, bitwise the same (no order of atomics),
    and against the oracle at the bounds of test_loss_and_gradient_match_oracle."""
    from paper_1806_10589_gb300 import WarmStartNet

    B, shape = 3, (500, 8, 16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert B * shape[0] // 2 > 4 * sms, "several planes per CTA on the coarse level too"
    rng = np.random.default_rng(4)
    masks = (rng.random((B,) + shape) < 0.35).astype(np.uint8)
    targets = rng.standard_normal((B, N.NOUT) + shape).astype(np.float32)
    p = _he(2, 32, 17)
    net = WarmStartNet(2, 32, stream=torch.cuda.current_stream())
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
        lb, gb = N.loss_and_grad(p.astype(np.float64), 1.0 - masks[b], targets[b], 2, 32)
        ref_loss += lb * nb / npore
        ref_g += gb * nb / npore
    assert abs(loss - ref_loss) <= 1e-2 * ref_loss, (loss, ref_loss)
    k = 0
    for li, (co, ci) in enumerate(N.layer_shapes(2, 32)):
        n = co * 27 * ci + co
        rel = np.linalg.norm(g[k:k + n] - ref_g[k:k + n]) / np.linalg.norm(ref_g[k:k + n])
        assert rel <= 0.06, (li, co, ci, rel)
        k += n

"""Convolutions of the warm-start network at the edges of their tiling (GB300),
against the FP64 oracle, with the bounds derived in test_gpu_wsnet.py: volumes of
one or two voxels a side, long rows, several patches and samples."""
import numpy as np
import pytest

from oracle import wsnet_oracle as N
from test_gpu_wsnet import _bf16, _padded, _unpad, torch  # noqa: F401

pytestmark = pytest.mark.gpu

PAIRS = [(32, 32), (32, 64), (64, 32), (64, 64), (128, 64)]
SHAPES = [(1, 1, 1, 1), (2, 2, 1, 3), (1, 2, 3, 260), (3, 5, 4, 66), (1, 9, 35, 16)]  # B, Z, Y, X


@pytest.mark.parametrize("cin,cout", PAIRS)
@pytest.mark.parametrize("shape", SHAPES)
def test_conv_shapes_match_oracle(torch, cin, cout, shape):  # noqa: F811
    from paper_1806_10589_gb300 import conv3d_bf16

    B, Z, Y, X = shape
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
        assert (np.abs(_unpad(out)[b] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), "forward"
        ref, rw, _ = N.conv_backward(a[b], w, g[b])
        S, sw, _ = N.conv_backward(np.abs(a[b]), np.abs(w), np.abs(g[b]))
        assert (np.abs(_unpad(gin)[b] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), "data gradient"
        ref_w, S_w = ref_w + rw, S_w + sw
    got = gw.double().cpu().numpy().transpose(0, 2, 1) - 0.5
    assert (np.abs(got - ref_w) <= 2.0 ** -16 * (S_w + 0.5)).all(), "weight gradient"

"""The choice between the two convolution kernels of the narrow layers (GB300)."""
import numpy as np
import pytest

from oracle import wsnet_oracle as N
from test_gpu_wsnet import _bf16, _padded, _unpad, torch  # noqa: F401

pytestmark = pytest.mark.gpu


# B, Z, Y, X.  Thin slabs, mostly border rows: every pair marches, with column changes
# inside a CTA (600 planes).  At 16^3 none does, at 40^3 32 -> 64 and 64 -> 32 do.
@pytest.mark.parametrize("cin,cout", [(32, 32), (32, 64), (64, 32), (64, 64)])
@pytest.mark.parametrize("shape", [(200, 3, 8, 14), (1, 16, 16, 16), (2, 40, 40, 40)])
def test_layers_on_both_sides_of_the_rule(torch, cin, cout, shape):  # noqa: F811
    """Against the FP64 oracle, bounds of test_gpu_wsnet.py."""
    from paper_1806_10589_gb300 import conv3d_bf16

    B, Z, Y, X = shape
    rng = np.random.default_rng(cin + 3 * cout + X)
    ta, a = _padded(torch, rng.standard_normal((B, cin, Z, Y, X)))
    tg, g = _padded(torch, rng.standard_normal((B, cout, Z, Y, X)))
    wb = _bf16(torch, rng.standard_normal((cout, 27, cin)) / np.sqrt(27 * cin))
    w = wb.double().numpy().transpose(0, 2, 1)
    tw = wb.cuda().contiguous()
    b64 = rng.standard_normal(cout)
    tb = torch.tensor(b64.astype(np.float32)).cuda()
    b64 = b64.astype(np.float32).astype(np.float64)
    st = torch.cuda.current_stream()
    out = torch.full((B, Z + 2, Y + 2, X + 2, cout), 7.0, dtype=torch.bfloat16, device="cuda")
    gin = torch.full((B, Z + 2, Y + 2, X + 2, cin), 7.0, dtype=torch.bfloat16, device="cuda")
    conv3d_bf16(0, ta.data_ptr(), 0, tw.data_ptr(), tb.data_ptr(), 1, out.data_ptr(), B, X, Y, Z, cin, cout, st)
    conv3d_bf16(1, tg.data_ptr(), 0, tw.data_ptr(), 0, 0, gin.data_ptr(), B, X, Y, Z, cin, cout, st)
    for t in (out, gin):
        border = t.clone()
        border[:, 1:-1, 1:-1, 1:-1, :] = 0
        assert not border.any(), "border rows must be written 0"
    out, gin = _unpad(out), _unpad(gin)
    flip = w.transpose(1, 0, 2)[:, :, ::-1]  # data gradient: transposed channels, taps reversed
    zero = np.zeros(cin)
    for b in range(0, B, max(1, B // 20)):
        ref, S = N.relu(N.conv(a[b], w, b64)), N.conv(np.abs(a[b]), np.abs(w), np.abs(b64))
        assert (np.abs(out[b] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), ("forward", b)
        ref, S = N.conv(g[b], flip, zero), N.conv(np.abs(g[b]), np.abs(flip), zero)
        assert (np.abs(gin[b] - ref) <= 2.0 ** -8 * np.abs(ref) + 2.0 ** -16 * S).all(), ("data gradient", b)


def test_small_narrow_layers_cost_no_more_than_wide_ones(torch):  # noqa: F811
    """24^3 voxels: a 32 -> 32 layer against the 32 -> 128 one, four times its work on
    the kernel that needs no resident weights, and 64 -> 64 against 64 -> 128."""
    from paper_1806_10589_gb300 import conv3d_bf16

    def us(cin, cout, n=24):
        st = torch.cuda.current_stream()
        x = torch.zeros((n + 2) ** 3 * cin, dtype=torch.bfloat16, device="cuda")
        y = torch.zeros((n + 2) ** 3 * cout, dtype=torch.bfloat16, device="cuda")
        w = torch.zeros(cout * 27 * cin, dtype=torch.bfloat16, device="cuda")
        return 1e3 * min(conv3d_bf16(0, x.data_ptr(), 0, w.data_ptr(), 0, 0, y.data_ptr(), 1, n, n, n, cin, cout, st,
                                     reps=100) for _ in range(5))

    times = [(us(32, 32), us(32, 128)), (us(64, 64), us(64, 128))]
    assert all(a <= 1.2 * b for a, b in times), times

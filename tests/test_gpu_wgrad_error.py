"""Error of the weight gradient of the narrow layers against 64 bits (GB300).

The tensor core truncates as it adds, so a sum's error grows with the products that
one accumulator takes: the kernel that marches along z takes no more than the one that
splits the rows, whose errors these bounds are (plus 10 %, the spread over seeds being
under 2 %).  With accumulators of 64 products throughout they were up to 1.6 times
as large (8 x 24^3, 32 -> 64: 5.8e-7; 1 x 20^3: 2.4e-7; 2 x 17x20x33: 4.2e-7)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (B, Z, Y, X), (cin, cout): relative error of the row-splitting kernel
BOUNDS = {((8, 24, 24, 24), (32, 32)): 3.80e-7, ((8, 24, 24, 24), (32, 64)): 3.70e-7,
          ((8, 24, 24, 24), (64, 32)): 3.69e-7, ((1, 48, 48, 48), (32, 64)): 3.74e-7,
          ((3, 30, 20, 60), (64, 64)): 4.99e-7, ((1, 20, 20, 20), (32, 32)): 1.72e-7,
          ((1, 20, 20, 20), (64, 32)): 1.69e-7, ((2, 17, 20, 33), (64, 64)): 2.20e-7,
          ((1, 64, 64, 64), (32, 32)): 6.39e-7, ((1, 64, 64, 64), (64, 32)): 6.46e-7,
          ((8, 72, 4, 72), (64, 32)): 4.18e-7, ((8, 72, 4, 72), (64, 64)): 6.34e-7,
          ((8, 40, 40, 40), (32, 64)): 1.25e-6, ((4, 36, 52, 44), (64, 64)): 1.66e-6}


@pytest.mark.parametrize("shape,pair", list(BOUNDS))
def test_weight_gradient_error(shape, pair):
    torch = pytest.importorskip("torch")
    from paper_1806_10589_gb300 import conv3d_bf16

    (B, Z, Y, X), (cin, cout) = shape, pair
    err = []
    for seed in range(3):
        gen = torch.Generator(device="cuda").manual_seed(seed)

        def rows(c, relu):
            t = torch.zeros(B, Z + 2, Y + 2, X + 2, c, device="cuda", dtype=torch.bfloat16)
            v = torch.randn(B, Z, Y, X, c, generator=gen, device="cuda")
            t[:, 1:-1, 1:-1, 1:-1] = (v.relu() if relu else 0.1 * v).bfloat16()
            return t

        a, g = rows(cin, True), rows(cout, False)
        out = torch.zeros(cout, 27, cin, device="cuda")
        conv3d_bf16(2, a.data_ptr(), g.data_ptr(), out.data_ptr(), 0, 0, out.data_ptr(), B, X, Y, Z, cin, cout,
                    torch.cuda.current_stream())
        g64 = g[:, 1:-1, 1:-1, 1:-1].double().reshape(-1, cout)
        ref = torch.stack([g64.t() @ a[:, z:z + Z, y:y + Y, x:x + X].double().reshape(-1, cin)
                           for z in range(3) for y in range(3) for x in range(3)], 1)
        err.append(float((out.double() - ref).norm() / ref.norm()))
    assert np.mean(err) <= 1.1 * BOUNDS[shape, pair], err

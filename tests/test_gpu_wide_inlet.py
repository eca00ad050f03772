"""Wide inlets (GB300).  A step leaves its parts of the inlet sum per warp, from 65,536
nodes on the planes z = 0 and z = 1 (FP64: 131,072) per 256-node tile, and from 524,288
nodes they are added to 128 behind the step."""
import numpy as np
import pytest

import oracle as O
from lbm_inputs import random_mask, uniform_field

pytestmark = pytest.mark.gpu


def _density_both_ways(shape, prec, variant):
    """(state, (flux, density)) from the parts of the steps, and with the plane's sum
    formed again before every step."""
    from paper_1806_10589_gb300 import Lattice

    mask = random_mask(*shape, 0.1, 7)
    f0 = O.W[:, None, None, None] * (1.05 + 0.01 * uniform_field((19,) + mask.shape, 3))

    def run(again):
        with Lattice(mask, 0.8, "mrt", prec) as lat:
            lat.set_kernel(variant)
            lat.set_flux_bc(0.5)
            lat.set_distributions(f0)
            for _ in range(6):
                if again:
                    lat.set_flux_bc(0.5)
                lat.step(1)
            return lat.distributions(), lat.get_flux()

    return run(False), run(True)


@pytest.mark.parametrize("shape", [(373, 390, 3), (701, 640, 4), (250, 260, 4)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-6)])
@pytest.mark.parametrize("variant", [0, 2, 3])
def test_wide_inlet_density(shape, prec, tol, variant):
    """On both sides of the second rule; the bounds of test_gpu_windows.py (at most 3e5 FP64
    terms below 0.1 in two orders: 1e-12 of the density)."""
    (a, fa), (b, fb) = _density_both_ways(shape, prec, variant)
    np.testing.assert_allclose(a, b, rtol=0, atol=tol)
    np.testing.assert_allclose(fa[1], fb[1], rtol=0, atol=tol)
    np.testing.assert_allclose(fa[0], fb[0], rtol=0, atol=tol * shape[0] * shape[1])


@pytest.mark.parametrize("shape", [(16, 16, 3), (31, 17, 4), (520, 530, 3), (611, 640, 3)])
@pytest.mark.parametrize("prec,ulp", [("fp16dev", 2.0 ** -15), ("bf16dev", 2.0 ** -12)])
@pytest.mark.parametrize("variant", [0, 3])
def test_inlet_density_of_16_bit_parts(shape, prec, ulp, variant):
    """The same in 16 bits.  Two-buffer: both densities are sums of the same stored
    values, 1e-6.  AA pattern: forming the plane's sum re-encodes the state, so values
    of about 0.05 differ by their rounding (ulp: theirs, over the weight) in every step,
    independently by node: 6 deviations of the mean of 6 steps.  One folded part left
    out would be more than 0.01 / 128."""
    (_, fa), (_, fb) = _density_both_ways(shape, prec, variant)
    a_in = 0.9 * shape[0] * shape[1]
    assert abs(fa[1] - 1.0) > 0.01
    assert abs(fa[1] - fb[1]) <= (1e-6 if variant == 0 else 36 * ulp / np.sqrt(a_in))


def test_step_cost_of_a_wide_inlet():
    """Time per step of an open 1024x1024x3 lattice, two thirds of whose nodes enter
    the inlet sum, against a 128x128x192 one of as many nodes: linear work, under 3
    times (1.7; 2.1 with one sum at the end of the step, 8.2 when every inlet block
    added a part per warp)."""
    import torch

    from paper_1806_10589_gb300 import Lattice

    def us(nx, ny, nz):
        st = torch.cuda.current_stream()
        with Lattice(np.zeros((nz, ny, nx), np.uint8), 0.8, "mrt", "fp32", stream=st) as lat:
            lat.set_flux_bc(1.0)
            lat.step(40)
            best = np.inf
            for _ in range(3):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(st)
                lat.step(80)
                b.record(st)
                b.synchronize()
                best = min(best, a.elapsed_time(b) / 80 * 1e3)
            return best

    wide, cube = us(1024, 1024, 3), us(128, 128, 192)
    assert wide <= 3 * cube, (wide, cube)

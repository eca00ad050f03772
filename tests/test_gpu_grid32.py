"""The step kernels without row windows (GB300): boxes and ensembles of 2^27 windows or
more take the id grid with 32-bit offsets.  Same values, same arithmetic as the
windows: bitwise equal states (ensembles large enough to take the windows; the 16-bit
forms compare one node per thread with two)."""
import numpy as np
import pytest

import oracle as O
from lbm_inputs import random_mask, uniform_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 5, 6), (31, 17, 9), (92, 2, 9)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("variant", [0, 3])
def test_lattice_without_windows(monkeypatch, shape, prec, variant):
    from paper_1806_10589_gb300 import Lattice

    mask = random_mask(*shape, 0.3, 11)
    f0 = O.W[:, None, None, None] * (1.0 + 0.01 * uniform_field((19,) + mask.shape, 3))

    def run():
        with Lattice(mask, 0.8, "mrt", prec) as lat:
            lat.set_kernel(variant)
            lat.set_flux_bc(0.002)
            lat.set_distributions(f0)
            lat.step(5)
            return lat.distributions()

    want = run()
    monkeypatch.setenv("GB300_LBM_NO_WINDOWS", "1")
    np.testing.assert_array_equal(run(), want)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16dev", "bf16dev"])
def test_large_ensemble_without_windows(monkeypatch, prec):
    from paper_1806_10589_gb300 import Batch

    masks = [random_mask(*s, 0.1, 5 + k) for k, s in enumerate([(61, 70, 75), (29, 31, 12), (90, 30, 24)])]

    def run():
        with Batch(masks, 0.8, "mrt", prec) as b:
            assert b.info()["n_tiles"] >= 1216
            for k in range(len(masks)):
                b.set_flux_bc(k, 0.05 * (k + 1))
            b.step(4)
            return [np.stack(b.fields(k)) for k in range(len(masks))]

    want = run()
    monkeypatch.setenv("GB300_LBM_NO_WINDOWS", "1")
    for a, b in zip(run(), want):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("shape", [(1, 6, 5), (31, 4, 3), (92, 3, 4)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_colour_without_windows(monkeypatch, shape, prec):
    from paper_1806_10589_gb300 import ColorLattice

    mask = random_mask(*shape, 0.3, 13)
    phi = np.where(uniform_field(mask.shape, 5) > 0, 0.75, -0.5)

    def run():
        with ColorLattice(mask, 0.8, 0.01, 0.9, -0.5, prec) as c:
            c.set_flux_bc(0.002, 1.0)
            c.set_phase(phi)
            c.step(6)
            return c.state()

    want = run()
    monkeypatch.setenv("GB300_LBM_NO_WINDOWS", "1")
    for a, b in zip(run(), want):
        np.testing.assert_array_equal(a, b)


def test_cost_without_windows(monkeypatch):
    """FP16 ensemble step without windows: under 0.95 of the 64-bit form's time (0.87
    measured; 1 when the ensembles without windows took that form)."""
    import torch

    from paper_1806_10589_gb300 import Batch

    masks = [random_mask(120, 110, 100, 0.4, k) for k in range(4)]
    monkeypatch.setenv("GB300_LBM_NO_WINDOWS", "1")

    def us():
        st = torch.cuda.current_stream()
        with Batch(masks, 0.8, "mrt", "fp16dev", stream=st) as b:
            b.step(50)
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            best = np.inf
            for _ in range(3):
                a.record(st)
                b.step(100)
                e.record(st)
                e.synchronize()
                best = min(best, a.elapsed_time(e) * 10)
            return best

    grid32 = us()
    monkeypatch.setenv("GB300_LBM_BATCH_ADDR64", "1")
    grid64 = us()
    assert grid32 <= 0.95 * grid64, (grid32, grid64)

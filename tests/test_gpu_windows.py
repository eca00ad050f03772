"""Row-window neighbour look-up of the step kernels against the id-grid form (GB300).

Both forms read the same values into the same arithmetic, so the states are
bitwise equal.  Widths around multiples of 30 put runs across window borders.
The 16-bit formats also compare two nodes per thread (windows) with one (id
grid): odd node counts, one to several 256-node tiles.
"""
import numpy as np
import pytest

import oracle as O
from lbm_inputs import random_mask, uniform_field

pytestmark = pytest.mark.gpu


def _state(mask, prec, variant, steps):
    from paper_1806_10589_gb300 import Lattice

    f0 = O.W[:, None, None, None] * (1.0 + 0.01 * uniform_field((19,) + mask.shape, 3))
    with Lattice(mask, 0.8, "mrt", prec) as lat:
        lat.set_kernel(variant)
        lat.set_flux_bc(0.002)
        lat.set_distributions(f0)
        lat.step(steps)
        return lat.distributions()


@pytest.mark.parametrize("shape", [(1, 5, 6), (29, 4, 5), (30, 4, 5), (31, 3, 7), (59, 4, 4), (60, 4, 4), (61, 5, 5),
                                   (90, 3, 4), (92, 2, 9)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("variant", [0, 3])
def test_windows_equal_id_grid(monkeypatch, shape, prec, variant):
    mask = random_mask(*shape, 0.3, 11)
    got = _state(mask, prec, variant, 5)
    monkeypatch.setenv("GB300_LBM_STEP_ADDR64", "1")
    monkeypatch.setenv("GB300_LBM_AA_ADDR64", "1")
    np.testing.assert_array_equal(got, _state(mask, prec, variant, 5))


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("config", [0, 1])
def test_large_ensemble_windows_equal_id_grid(monkeypatch, prec, config):
    """Ensembles of 1216 tiles or more take the row windows (16-bit: two nodes per
    thread); odd pore counts, members of one and of many windows per row."""
    from paper_1806_10589_gb300 import Batch

    masks = [random_mask(*s, 0.1, 5 + k) for k, s in enumerate([(61, 70, 75), (29, 31, 12), (90, 30, 24)])]

    def run():
        with Batch(masks, 0.8, "mrt", prec) as b:
            b.set_config(config)
            assert b.info()["n_tiles"] >= 1216
            for k in range(len(masks)):
                b.set_flux_bc(k, 0.05 * (k + 1))
            b.step(4)
            return [np.stack(b.fields(k)) for k in range(len(masks))], [b.get_flux(k) for k in range(len(masks))]

    got = run()
    monkeypatch.setenv("GB300_LBM_BATCH_ADDR64", "1")
    want = run()
    for a, b in zip(got[0], want[0]):
        np.testing.assert_array_equal(a, b)
    assert got[1] == want[1]


@pytest.mark.parametrize("shape", [(4, 3, 3), (16, 16, 3), (31, 17, 4), (70, 61, 5)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-6)])
@pytest.mark.parametrize("variant", [0, 1, 2, 3])
def test_inlet_density_of_parts_equals_the_plane_sum(shape, prec, tol, variant):
    """The inlet density from the parts a step leaves, against the sum over the inlet
    plane that setting the flux again forms before each step (one part to several
    tiles of parts, inlet blocks with and without slots past the last node).  Sums of
    at most 1.3e4 FP64 terms below 0.1 in two orders: 1e-13; FP32 values: one rounding
    of the density more or less."""
    from paper_1806_10589_gb300 import Lattice

    mask = random_mask(*shape, 0.2, 7)
    f0 = O.W[:, None, None, None] * (1.0 + 0.01 * uniform_field((19,) + mask.shape, 3))

    def run(again):
        with Lattice(mask, 0.8, "mrt", prec) as lat:
            lat.set_kernel(variant)
            lat.set_flux_bc(0.002)
            lat.set_distributions(f0)
            for _ in range(3):
                if again:
                    for _ in range(2):
                        lat.set_flux_bc(0.002)
                        lat.step(1)
                else:
                    lat.step(2)
            return lat.distributions(), lat.get_flux()

    (a, fa), (b, fb) = run(False), run(True)
    np.testing.assert_allclose(a, b, rtol=0, atol=tol)
    np.testing.assert_allclose(fa, fb, rtol=0, atol=tol * mask.shape[1] * mask.shape[2])


@pytest.mark.parametrize("shape", [(1, 6, 5), (30, 1, 4), (31, 4, 3), (61, 5, 5), (92, 3, 4)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_colour_windows_equal_id_grid(monkeypatch, shape, prec):
    """Colour step on the row windows and face bits against the id grid: boxes of one
    voxel across, pores on every face and edge, runs across window borders."""
    from paper_1806_10589_gb300 import ColorLattice

    mask = random_mask(*shape, 0.3, 13)
    phi = np.where(uniform_field(mask.shape, 5) > 0, 0.75, -0.5)

    def run():
        with ColorLattice(mask, 0.8, 0.01, 0.9, -0.5, prec) as c:
            c.set_flux_bc(0.002, 1.0)
            c.set_phase(phi)
            c.step(6)
            return c.state()

    got = run()
    monkeypatch.setenv("GB300_LBM_COLOR_ADDR64", "1")
    for a, b in zip(got, run()):
        np.testing.assert_array_equal(a, b)

"""Inlet density that a step in pressure mode records (GB300): the one the prescribed
flux would need, as lbm_get_flux reports it once the inlet is back in flux mode."""
import numpy as np
import pytest

import oracle as O
from lbm_inputs import random_mask, uniform_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-6), ("fp16dev", 1e-5)])
@pytest.mark.parametrize("variant", [0, 1, 2, 3])
def test_density_after_pressure_mode(prec, tol, variant):
    """Against the sum over the inlet plane of the state that the last step in pressure
    mode read (FP64: two summation orders; 16 bits: the part is formed from the rounded
    values: weights that add to 1 times half an ulp of a deviation of order 0.01, 4e-6)."""
    import torch

    from paper_1806_10589_gb300 import Lattice

    mask = random_mask(9, 7, 12, 0.2, 3)
    f0 = O.W[:, None, None, None] * (1.0 + 0.01 * uniform_field((19,) + mask.shape, 3))
    want = torch.zeros(1, dtype=torch.float64, device="cuda")
    with Lattice(mask, 0.8, "mrt", prec, stream=torch.cuda.current_stream()) as lat:
        lat.set_kernel(variant)
        lat.set_flux_bc(0.01)
        lat.set_distributions(f0)
        lat.step(3)
        before = lat.get_flux()[1]
        lat.set_pressure_bc(4, 1.01)
        for _ in range(2):  # both inlet-density slots
            lat.step(3)
            lat.inlet_density_noalloc(want.data_ptr())
            lat.step(1)
            assert lat.get_flux()[1] == 1.01
        lat.set_flux_bc(0.02)
        got = lat.get_flux()[1]
        assert abs(got - float(want)) <= tol, (got, float(want), before)
        assert abs(got - before) > 10 * tol, "not the density recorded before the pressure steps"

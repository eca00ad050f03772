"""Error of an FP64 run against extended precision (GB300).

The collision's constants are rounded once.  Where their sum over the directions is
not 1 to that accuracy, every step multiplies the density by the same factor and the
error grows with the steps instead of their square root."""
import numpy as np
import pytest

import oracle as O
from lbm_inputs import random_mask, uniform_field

pytestmark = pytest.mark.gpu

LD = np.longdouble
XI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]
W = [LD(1) / 3] + [LD(1) / 18] * 6 + [LD(1) / 36] * 12


def _run(mask, d, sp, sm, Q, drho_out, steps):
    """The step of the library on shifted distributions d[q][node], extended precision."""
    nz, ny, nx = mask.shape
    grid = np.full((nz + 2, ny + 2, nx + 2), -1)
    pore = mask == 0
    n = int(pore.sum())
    grid[1:-1, 1:-1, 1:-1][pore] = np.arange(n)
    z, y, x = np.nonzero(np.pad(pore, 1))
    src = [grid[z - c[2], y - c[1], x - c[0]] for c in XI]
    inl, out = z == 1, z == nz
    c = np.array(XI)

    def close(e, s, uz):
        tx = LD(0.5) * (e[1] + e[7] + e[9] - e[2] - e[10] - e[8])
        ty = LD(0.5) * (e[3] + e[7] + e[10] - e[4] - e[9] - e[8])
        for a, b, t in ((5, 6, 0), (11, 12, -tx), (14, 13, tx), (15, 16, -ty), (18, 17, ty)):
            if s > 0:
                e[a] = e[b] + uz / (3 if a == 5 else 6) + t
            else:
                e[b] = e[a] - uz / (3 if a == 5 else 6) - t

    for _ in range(steps):
        e = np.stack([d[0]] + [np.where(src[q] >= 0, d[q][src[q]], d[OPP[q]]) for q in range(1, 19)])
        flat = e[[0, 1, 2, 3, 4, 7, 8, 9, 10]].sum(0)
        k_in, k_out = flat + 2 * e[[6, 12, 13, 16, 17]].sum(0), flat + 2 * e[[5, 11, 14, 15, 18]].sum(0)
        drho_in = (LD(Q) + k_in[inl].sum()) / int(inl.sum())
        a, b = e[:, inl], e[:, out]
        close(a, 1, drho_in - k_in[inl])
        close(b, -1, k_out[out] - LD(drho_out))
        e[:, inl], e[:, out] = a, b
        drho = e.sum(0)
        u = [sum(int(v) * e[q] for q, v in enumerate(c[:, k]) if v) for k in range(3)]
        uu = LD(1.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
        d = e.copy()
        d[0] = e[0] - sp * (e[0] - W[0] * (drho - uu))
        for q in range(1, 19):
            xu = sum(int(v) * w for v, w in zip(XI[q], u) if v)
            p = LD(0.5) * (e[q] + e[OPP[q]]) - W[q] * (drho + LD(4.5) * xu * xu - uu)
            m = LD(0.5) * (e[q] - e[OPP[q]]) - 3 * W[q] * xu
            d[q] = e[q] - sp * p - sm * m
    return d


@pytest.mark.parametrize("tau", [0.7, 1.0])
@pytest.mark.parametrize("variant", [0, 3])
def test_fp64_run_against_extended_precision(tau, variant):
    """Relative error of the distributions after 150 steps: at most 2^-54 a step from
    the constants (the only rounded one in their sum, s+ / 3 < 1/2, is off by 2^-55 at most)
    and a random walk of 2^-53 a step from the operations; reading f = w + d back
    rounds each value once."""
    from paper_1806_10589_gb300 import Lattice

    steps, Q = 150, 1e-3
    mask = random_mask(8, 7, 26, 0.15, 4)
    f0 = O.W[:, None, None, None] * (2.0 + 0.01 * uniform_field((19,) + mask.shape, 3))
    with Lattice(mask, tau, "mrt", "fp64") as lat:
        lat.set_kernel(variant)
        lat.set_flux_bc(Q)
        lat.set_pressure_bc(5, 2.0)
        lat.set_distributions(f0)
        lat.step(steps)
        got = lat.distributions()
    pore = mask == 0
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None]
    sp = 1.0 / tau
    ref = _run(mask, (f0[:, pore] - w).astype(LD), LD(sp), LD(8.0 * (2.0 - sp) / (8.0 - sp)), Q, 1.0, steps)
    err = got[:, pore].astype(LD) - w.astype(LD) - ref
    rel = float(np.sqrt((err * err).sum() / (ref * ref).sum()))
    assert rel <= steps * 2.0 ** -54 + (np.sqrt(steps) + 2) * 2.0 ** -53, rel

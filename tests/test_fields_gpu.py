"""Initial states, output fields and reductions against the FP64 oracle and
numpy: both CTA sizes, walls and masks, one cell, remainders."""
import numpy as np
import pytest

import oracle
from _helpers import direction_map, gpu_run, oracle_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 6, 37), (5, 7, 9), (61, 65, 70)]
STORAGES = {"f32": 6e-8, "f64": 1.2e-16, "f16_dev": 2.0 ** -11, "bf16_dev": 2.0 ** -8, "f16_rel": 2.0 ** -11,
            "bf16_rel": 2.0 ** -8}


def _setup(shape, geometry):
    r1, r2, u = wl.random_state(shape, seed=5, rho_lo=0.3, rho_hi=0.7, u_max=0.04)
    kw, solid = {}, None
    if geometry == "walls":
        kw = dict(periodic=(1, 1, 0), rho_s=(0.02, 0.05))
    elif geometry == "mask":
        solid = np.zeros(shape, dtype=np.uint8)
        solid[0, : (shape[1] + 1) // 2, ::3] = 1
        if solid.all():
            solid[...] = 0
        u[solid != 0] = 0.0
        kw = dict(rho_s=(0.02, 0.05))
    return r1, r2, u, solid, kw


@pytest.mark.parametrize("storage", list(STORAGES))
@pytest.mark.parametrize("geometry", ["periodic", "walls", "mask"])
@pytest.mark.parametrize("moving", [False, True])
def test_initial_populations(gpu_lib, storage, geometry, moving):
    """f_i = f^eq_i(rho, u): rounded once in FP32 and FP64; the 16-bit formats
    round the deviation (at most 0.45 of the population's scale here)."""
    perm = direction_map()
    for shape in SHAPES:
        r1, r2, u, solid, kw = _setup(shape, geometry)
        _, f = oracle_run(shape, r1, r2, u if moving else None, 0, G12=-1.0, solid=solid, **kw)
        extra = {"rho0_dev": 0.5} if storage.endswith("_dev") else {}
        lat = gpu_run(shape, r1, r2, u if moving else None, 0, storage=storage, G12=-1.0, solid=solid, **kw, **extra)
        g = lat.get_populations()
        lat.close()
        ref = f[:, perm]
        if solid is not None:
            ref = np.where(solid[None, None] != 0, 0.0, ref)
        tol = STORAGES[storage] * np.abs(ref).max() * (4 if storage == "f64" else 2)
        assert np.abs(g - ref).max() < tol, shape


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("geometry", ["periodic", "walls", "mask"])
@pytest.mark.parametrize("out_f64", [False, True])
def test_fields_and_reductions(gpu_lib, storage, geometry, out_f64):
    """rho^a sum 19 terms, u_F some 60 more: 80 roundings of the values' scale."""
    for shape in SHAPES:
        r1, r2, u, solid, kw = _setup(shape, geometry)
        p, f = oracle_run(shape, r1, r2, u, 1, G12=-1.0, tau=(0.8, 1.1), solid=solid, **kw)
        a, b, uF = oracle.moments(p, f)
        fluid = np.ones(shape, bool) if solid is None else solid == 0
        a, b, uF = (np.where(fluid, a, 0), np.where(fluid, b, 0), np.where(fluid[..., None], uF, 0))
        lat = gpu_run(shape, r1, r2, u, 1, storage=storage, G12=-1.0, tau=(0.8, 1.1), solid=solid, **kw)
        ga, gb, guF = lat.moments(out_f64=out_f64)
        red = lat.reduce()
        lat.close()
        eps = 80 * (6e-8 if storage == "f32" or not out_f64 else 1.2e-16)
        assert np.abs(ga - a).max() < eps and np.abs(gb - b).max() < eps and np.abs(guF - uF).max() < eps
        eps = 80 * STORAGES[storage]
        n = fluid.sum()
        assert abs(red["mass1"] - a.sum()) < eps * n and abs(red["mass2"] - b.sum()) < eps * n
        assert np.abs(np.array(red["momentum"]) - ((a + b)[..., None] * uF).sum((0, 1, 2))).max() < eps * n
        assert abs(red["max_uF"] - np.sqrt((uF ** 2).sum(-1)).max()) < eps


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("centre,r_in,r_out", [((10.0, 8.0, 6.0), 5.0, 5.0), ((10.5, 8.5, 6.5), 6.5, 9.0),
                                               ((0.3, 21.7, 3.1), 4.2, 7.9), ((10.0, 8.0, 6.0), 13.0, 13.0)])
def test_pressure_regions(gpu_lib, storage, centre, r_in, r_out):
    """Whole radii put cells exactly on the spheres: the regions are those of the
    FP64 distance, cell for cell (equal means up to FP64 summation)."""
    shape = (24, 26, 28)
    r1, r2, _, _, _ = _setup(shape, "periodic")
    lat = gpu_run(shape, r1, r2, None, 1, storage=storage, G12=-1.2)
    a, b, _ = lat.moments(out_f64=True)
    got = lat.pressure_jump(centre, r_in, r_out)
    lat.close()
    z, y, x = np.meshgrid(*[np.arange(n, dtype=np.float64) for n in shape], indexing="ij")
    d2 = 0.0
    for v, c, n in ((x, centre[0], 28), (y, centre[1], 26), (z, centre[2], 24)):
        d = v - c
        d = np.where(d > 0.5 * n, d - n, np.where(d < -0.5 * n, d + n, d))
        d2 = d2 + d * d
    r = np.sqrt(d2)
    p = (a + b) / 3.0 + 1.2 / 3.0 * a * b
    # the densities of the fields and of the diagnostics are two orders of the
    # same 19-term sums
    tol = 40 * STORAGES[storage]
    assert abs(got[0] - p[r < r_in].mean()) < tol
    assert abs(got[1] - p[r > r_out].mean()) < tol

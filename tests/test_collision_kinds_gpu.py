"""The collision instances of the fused step that keep moments (or, at tau = 1,
nothing) of the populations instead of the populations themselves, against the
FP64 oracle, on tiles with remainders, z walls and a solid mask."""
import numpy as np
import pytest

from _helpers import direction_map, gpu_run, oracle_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# one cell, a full tile, one past a tile in x and y, chunks of z with a remainder
SHAPES = [(1, 1, 1), (3, 8, 32), (9, 9, 33), (19, 5, 70)]
# four steps of about 20 dependent FP32 roundings (6e-8 each) per population,
# relative to the largest population
TOL = 4 * 20 * 6e-8


def _geometry(kind, shape):
    if kind == "walls":
        return dict(periodic=(1, 1, 0), rho_s=(0.02, 0.05)), None
    if kind == "mask":
        solid = np.zeros(shape, dtype=np.uint8)
        solid[0, : (shape[1] + 1) // 2, ::3] = 1
        if solid.all():
            solid[...] = 0
        return dict(rho_s=(0.02, 0.05)), solid
    return {}, None


@pytest.mark.parametrize("forcing", ["edm", "guo"])
@pytest.mark.parametrize("collision,tau", [("bgk", (1.0, 1.0)), ("regularized", (0.7, 1.2)),
                                           ("regularized3", (0.8, 0.9)), ("bgk", (1.0, 0.8))])
@pytest.mark.parametrize("kind", ["periodic", "walls", "mask"])
@pytest.mark.parametrize("shape", SHAPES)
def test_instances_against_oracle(gpu_lib, shape, kind, collision, tau, forcing):
    perm = direction_map()
    geo, solid = _geometry(kind, shape)
    r1, r2, u = wl.random_state(shape, seed=7, rho_lo=0.3, rho_hi=0.7, u_max=0.03)
    if solid is not None:
        u[solid != 0] = 0.0
    kw = dict(tau=tau, G12=-1.2, G21=-1.1, g_ext=(1e-4, -2e-4, 5e-5), collision=collision, forcing=forcing, **geo)
    _, f = oracle_run(shape, r1, r2, u, 4, solid=solid, **kw)
    lat = gpu_run(shape, r1, r2, u, 4, storage="f32", solid=solid, **kw)
    g = lat.get_populations()
    lat.close()
    ref = f[:, perm]
    if solid is not None:
        ref = np.where(solid[None, None] != 0, 0.0, ref)
    assert np.abs(g - ref).max() < TOL * np.abs(ref).max()


@pytest.mark.parametrize("storage", ["f32", "f16_dev"])
@pytest.mark.parametrize("forcing", ["edm", "guo"])
def test_operators_coincide_at_tau_one(gpu_lib, storage, forcing):
    """tau = 1 in both components: the three operators are one step, bit for bit."""
    shape = (9, 9, 33)
    r1, r2, u = wl.random_state(shape, seed=3, rho_lo=0.4, rho_hi=0.6, u_max=0.02)
    got = []
    for collision in ("bgk", "regularized", "regularized3"):
        lat = gpu_run(shape, r1, r2, u, 3, storage=storage, G12=-1.2, collision=collision, forcing=forcing,
                      **({"rho0_dev": 0.5} if storage == "f16_dev" else {}))
        got.append(lat.get_populations())
        lat.close()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])

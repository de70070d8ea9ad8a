"""Runs of steps in moment space against the FP64 oracle: every tile of the step
kernel, with its remainders along all axes."""
import numpy as np
import pytest

from _helpers import direction_map, gpu_run, oracle_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# 20 dependent roundings per step and population, relative to the largest one
EPS = 20 * 6.0e-8
# tiles of 12, 16 and 24 rows at tau = 1, of 12, 16 and 16 regularized
TILES = [(27, 58, 147), (8, 285, 153), (10, 254, 99)]
KINDS = [("bgk", (1.0, 1.0)), ("regularized", (0.7, 1.2))]


def _compare(shape, collision, tau, calls, solid=None, storage="f32", tol=None, **geo):
    r1, r2, u = wl.random_state(shape, seed=11, rho_lo=0.3, rho_hi=0.7, u_max=0.03)
    if solid is not None:
        u[solid != 0] = 0.0
    kw = dict(tau=tau, G12=-1.2, G21=-1.1, g_ext=(1e-4, -2e-4, 5e-5), collision=collision, **geo)
    _, f = oracle_run(shape, r1, r2, u, sum(calls), solid=solid, **kw)
    lat = gpu_run(shape, r1, r2, u, 0, solid=solid, storage=storage, **kw)
    for n in calls:
        lat.step(n)
    g = lat.get_populations()
    lat.close()
    ref = f[:, direction_map()]
    if solid is not None:
        ref = np.where(solid[None, None] != 0, 0.0, ref)
    assert np.abs(g - ref).max() < (tol or sum(calls) * EPS * np.abs(ref).max())


@pytest.mark.parametrize("geometry", ["periodic", "mirror"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("shape", TILES)
def test_tiles(gpu_lib, shape, collision, tau, geometry):
    geo = {} if geometry == "periodic" else dict(rho_s=(0.02, 0.05), wall_model=geometry, periodic=(1, 1, 0))
    _compare(shape, collision, tau, [3], **geo)


def _scattered(shape):
    """One site in twelve solid, and a slab across the lattice."""
    solid = (np.random.default_rng(5).random(shape) < 1 / 12).astype(np.uint8)
    z, x = np.arange(shape[0])[:, None, None], np.arange(shape[2])[None, None, :]
    solid[np.broadcast_to((z + x // 2) % max(shape[0], 9) < 3, shape)] = 1
    return solid


@pytest.mark.parametrize("model", ["mirror", "potential"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("shape,calls", [(s, [4]) for s in TILES] + [((61, 65, 70), [2, 1, 3]), ((2, 200, 200), [3])])
def test_masks(gpu_lib, shape, collision, tau, model, calls):
    _compare(shape, collision, tau, calls, solid=_scattered(shape), rho_s=(0.02, 0.05), wall_model=model)


@pytest.mark.parametrize("geometry", ["periodic", "mirror", "mask"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("storage,eps,vmax", [("f16_dev", 2.0 ** -11, 0.4 / 3), ("bf16_dev", 2.0 ** -8, 0.4 / 3)])
@pytest.mark.parametrize("calls", [[2], [3], [4, 1, 3]])
def test_16_bit_formats(gpu_lib, storage, eps, vmax, collision, tau, geometry, calls):
    """A run rounds what it stores (at most vmax) once going in and once coming out:
    no further off than steps that do so each time, five such roundings a step (the
    collision mixes the incoming ones with weights that sum to at most about 4)."""
    shape = (61, 65, 70)
    geo = dict(periodic={}, mirror=dict(rho_s=(0.02, 0.05), wall_model="mirror", periodic=(1, 1, 0)),
               mask=dict(rho_s=(0.02, 0.05), wall_model="mirror", solid=_scattered(shape)))[geometry]
    _compare(shape, collision, tau, calls, storage=storage, tol=sum(calls) * 5 * eps * vmax, rho0_dev=0.5, **geo)


@pytest.mark.parametrize("geometry", ["periodic", "mirror", "mask"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("storage", ["f32", "f16_dev"])
@pytest.mark.parametrize("shape,calls", [(TILES[0], [3]), ((61, 65, 70), [2, 1, 6])])
def test_guo_forcing(gpu_lib, shape, calls, storage, collision, tau, geometry):
    geo = dict(periodic={}, mirror=dict(rho_s=(0.02, 0.05), wall_model="mirror", periodic=(1, 1, 0)),
               mask=dict(rho_s=(0.02, 0.05), wall_model="mirror", solid=_scattered(shape)))[geometry]
    if storage == "f16_dev":
        geo["rho0_dev"] = 0.5
    tol = None if storage == "f32" else sum(calls) * 5 * 2.0 ** -11 / 3
    _compare(shape, collision, tau, calls, storage=storage, tol=tol, forcing="guo", **geo)

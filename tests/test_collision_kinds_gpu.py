"""The step's kernels by collision kind, geometry, forcing and format against
the FP64 oracle: the marching kernel (lattices large enough for it, a call per
step), runs in moment space (the same lattices, several steps per call), the
box kernel of small and thin lattices, and the half-cell FP64 kernels."""
import numpy as np
import pytest

from _helpers import direction_map, gpu_run, oracle_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# box kernel: one cell, one box, remainders along every axis, one layer along
# y or z, columns; marching kernel and moment runs: tile and chunk remainders,
# fewer planes than a chunk's overlap
SMALL = [(1, 1, 1), (1, 9, 17), (1, 1, 40), (9, 1, 17), (4, 8, 8), (7, 9, 11), (13, 2, 3), (2, 5, 70)]
MARCH = [(61, 65, 70), (2, 200, 200), (3, 47, 900)]
KINDS = [("bgk", (1.0, 1.0)), ("regularized", (0.7, 1.2)), ("regularized3", (0.8, 0.9)), ("bgk", (1.0, 0.8))]
GEOMETRY = ["periodic", "mirror", "potential", "mask_mirror", "mask_potential"]
# four steps of about 20 dependent roundings per population, relative to the
# largest population
TOL = {"f32": 4 * 20 * 6.0e-8, "f64": 4 * 20 * 1.2e-16}


def _geometry(kind, shape):
    if kind == "periodic":
        return {}, None
    kw = dict(rho_s=(0.02, 0.05), wall_model=kind.split("_")[-1])
    if not kind.startswith("mask"):
        return dict(kw, periodic=(1, 1, 0)), None
    solid = np.zeros(shape, dtype=np.uint8)
    solid[0, : (shape[1] + 1) // 2, ::3] = 1
    solid[-1, :, shape[2] // 2:shape[2] // 2 + 2] = 1
    if solid.all():
        solid[...] = 0
    return kw, solid


def _compare(shape, geometry, collision, tau, forcing, storage, steps, tol, calls=None, **extra):
    perm = direction_map()
    geo, solid = _geometry(geometry, shape)
    r1, r2, u = wl.random_state(shape, seed=7, rho_lo=0.3, rho_hi=0.7, u_max=0.03)
    if solid is not None:
        u[solid != 0] = 0.0
    kw = dict(tau=tau, G12=-1.2, G21=-1.1, g_ext=(1e-4, -2e-4, 5e-5), collision=collision, forcing=forcing, **geo)
    _, f = oracle_run(shape, r1, r2, u, steps, solid=solid, **kw)
    lat = gpu_run(shape, r1, r2, u, 0, storage=storage, solid=solid, **kw, **extra)
    for n in calls or [steps]:
        lat.step(n)
    assert lat.step_count() == steps
    g = lat.get_populations()
    lat.close()
    ref = f[:, perm]
    if solid is not None:
        ref = np.where(solid[None, None] != 0, 0.0, ref)
    assert np.abs(g - ref).max() < tol(ref)


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("forcing", ["edm", "guo"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("geometry", GEOMETRY)
def test_small_and_thin_against_oracle(gpu_lib, geometry, collision, tau, forcing, storage):
    for shape in SMALL:
        _compare(shape, geometry, collision, tau, forcing, storage, 4, lambda ref: TOL[storage] * np.abs(ref).max())


@pytest.mark.parametrize("forcing", ["edm", "guo"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("geometry", ["periodic", "mirror", "mask_mirror"])
@pytest.mark.parametrize("shape", MARCH)
def test_marching_against_oracle(gpu_lib, shape, geometry, collision, tau, forcing):
    _compare(shape, geometry, collision, tau, forcing, "f32", 4, lambda ref: TOL["f32"] * np.abs(ref).max(),
             calls=[1, 1, 1, 1])


@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("geometry,shape", [(g, s) for g in ("periodic", "mirror", "potential") for s in MARCH] +
                         [("mirror", (1, 150, 300)), ("potential", (1, 150, 300))])
@pytest.mark.parametrize("calls", [[4], [2, 1, 3], [5]])
def test_runs_of_steps_against_oracle(gpu_lib, geometry, shape, collision, tau, calls):
    n = sum(calls)
    _compare(shape, geometry, collision, tau, "edm", "f32", n, lambda ref: n / 4 * TOL["f32"] * np.abs(ref).max(),
             calls=calls)


@pytest.mark.parametrize("storage,eps", [("f16_dev", 2.0 ** -11), ("bf16_dev", 2.0 ** -8)])
@pytest.mark.parametrize("forcing", ["edm", "guo"])
@pytest.mark.parametrize("collision,tau", KINDS)
@pytest.mark.parametrize("geometry", ["periodic", "mirror", "mask_mirror"])
@pytest.mark.parametrize("shape", [(1, 9, 17), (7, 9, 11), MARCH[0]])
def test_deviation_formats_one_step(gpu_lib, shape, geometry, collision, tau, forcing, storage, eps):
    """One step: the deviations are rounded once going in and once coming out
    (eps of the largest of them, 0.3 of 1/3 here); the collision mixes the 19
    incoming roundings with weights that sum to at most about 4."""
    dmax = 0.4 / 3.0
    _compare(shape, geometry, collision, tau, forcing, storage, 1, lambda ref: (4 + 1) * eps * dmax, rho0_dev=0.5)


@pytest.mark.parametrize("shape", [(9, 9, 33), MARCH[0]])
@pytest.mark.parametrize("storage", ["f32", "f16_dev", "f64"])
@pytest.mark.parametrize("forcing", ["edm", "guo"])
def test_operators_coincide_at_tau_one(gpu_lib, shape, storage, forcing):
    """tau = 1 in both components: the three operators are one step, bit for bit."""
    r1, r2, u = wl.random_state(shape, seed=3, rho_lo=0.4, rho_hi=0.6, u_max=0.02)
    got = []
    for collision in ("bgk", "regularized", "regularized3"):
        lat = gpu_run(shape, r1, r2, u, 3, storage=storage, G12=-1.2, collision=collision, forcing=forcing,
                      **({"rho0_dev": 0.5} if storage == "f16_dev" else {}))
        got.append(lat.get_populations())
        lat.close()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])

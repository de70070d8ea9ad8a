"""Runs of steps on lattices of few planes and on tall ones: which steps they take, and
that those are right beyond the lattices of the box step."""
import numpy as np
import pytest

from _helpers import direction_map, gpu_run, oracle_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

EQ, REG = ("bgk", 1.0), ("regularized", 0.7)


@pytest.mark.parametrize("shape,storage,kind,moments", [
    ((1, 2100, 2100), "f32", REG, False), ((2, 2100, 2100), "f32", REG, False), ((20000, 32, 32), "f32", REG, False),
    ((1, 4096, 4096), "f16_dev", EQ, False), ((2, 2100, 2100), "bf16_dev", REG, False), ((20000, 32, 32), "f16_dev", EQ, False),
    ((6, 2100, 2100), "f32", EQ, True), ((12, 1000, 1000), "f32", REG, True), ((24, 500, 500), "f16_dev", EQ, True),
    ((128, 128, 128), "f32", REG, True), ((128, 128, 128), "f16_dev", REG, True)])
def test_route(gpu_lib, shape, storage, kind, moments):
    """Twenty steps in one call run in moment space only where that is the faster way by
    a tenth or more either way, as measured step by step and in moment space."""
    from paper_1601_01237_gb300 import Lattice
    kw = dict(rho0_dev=0.5) if storage.endswith("_dev") else {}
    lat = Lattice(shape, storage=storage, collision=kind[0], tau=(kind[1],) * 2, **kw)
    names = set(lat.step_timed(20))
    lat.close()
    assert names == ({"k_moment_in", "k_step_moment", "k_moment_out"} if moments else {"k_step_fused"})


@pytest.mark.parametrize("shape", [(1, 2053, 2071), (3, 700, 803)])
@pytest.mark.parametrize("kind", [EQ, REG])
def test_few_planes(gpu_lib, shape, kind):
    """20 dependent roundings per step and population, relative to the largest one."""
    r1, r2, u = wl.random_state(shape, seed=12, rho_lo=0.3, rho_hi=0.7, u_max=0.03)
    kw = dict(tau=(kind[1],) * 2, G12=-1.2, G21=-1.1, collision=kind[0])
    _, f = oracle_run(shape, r1, r2, u, 3, **kw)
    lat = gpu_run(shape, r1, r2, u, 3, storage="f32", **kw)
    g = lat.get_populations()
    lat.close()
    ref = f[:, direction_map()]
    assert np.abs(g - ref).max() < 3 * 20 * 6.0e-8 * np.abs(ref).max()

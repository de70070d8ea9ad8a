"""Recordings of one shape share their memory: what a lattice recorded before
must not show in its gradients."""
import numpy as np
import pytest

from _helpers import gpu_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _gradient(lat, state, steps, every):
    lat.init_fields(*state)
    lat.record(steps, every)
    a, b, _ = lat.moments()
    d1, d2 = np.empty(a.shape), np.empty(a.shape)
    par = lat.adjoint(2 * a, b - 0.3, d1, d2)
    return d1, d2, np.array(par)


@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_recordings_in_a_row(gpu_lib, storage):
    """Same shape, another number of checkpoints, another segment length and back."""
    shape = (9, 10, 33)
    states = [wl.random_state(shape, seed=s, rho_lo=0.4, rho_hi=0.6, u_max=0.0)[:2] for s in (1, 2)]
    kw = dict(storage=storage, G12=-1.2)
    lat = gpu_run(shape, *states[0], None, 0, **kw)
    for steps, every, s in [(8, 4, 0), (8, 4, 1), (7, 4, 0), (7, 3, 1), (12, 3, 0), (3, 8, 1), (8, 4, 1)]:
        got = _gradient(lat, states[s], steps, every)
        fresh = gpu_run(shape, *states[s], None, 0, **kw)
        want = _gradient(fresh, states[s], steps, every)
        fresh.close()
        assert all(np.array_equal(g, w) for g, w in zip(got, want))
    lat.close()


@pytest.mark.parametrize("collision", ["bgk", "regularized", "regularized3"])
@pytest.mark.parametrize("geometry", ["periodic", "mirror", "mask_mirror"])
def test_reverse_step_of_tau_one(gpu_lib, collision, geometry):
    """FP32 at tau = 1 against the FP64 reverse pass, which sums the general form: 20
    dependent roundings a step, relative to the largest value."""
    shape, steps = (10, 12, 35), 12
    state = wl.random_state(shape, seed=3, rho_lo=0.4, rho_hi=0.6, u_max=0.0)[:2]
    kw = dict(G12=-1.2, G21=-1.1, g_ext=(1e-4, -2e-4, 5e-5), collision=collision, rho_s=(0.02, 0.05))
    solid = None
    if geometry == "mirror":
        kw.update(periodic=(1, 1, 0), wall_model="mirror")
    elif geometry == "mask_mirror":
        kw.update(wall_model="mirror")
        solid = np.zeros(shape, np.uint8)
        solid[:2, :, ::2] = 1
        solid[5:7, 3:9, 10:20] = 1
    got = []
    for storage in ("f32", "f64"):
        lat = gpu_run(shape, *state, None, 0, storage=storage, solid=solid, **kw)
        got.append(_gradient(lat, state, steps, 5))
        lat.close()
    for g, w in zip(*got):
        assert np.abs(g - w).max() < steps * 20 * 6.0e-8 * np.abs(w).max()

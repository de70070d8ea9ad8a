"""A recording takes the steps that the reverse pass recomputes."""
import numpy as np
import pytest

from _helpers import gpu_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f64", "f32", "f16_dev", "bf16_dev", "f16_rel"])
@pytest.mark.parametrize("collision,tau", [("bgk", 1.0), ("regularized", 0.7), ("regularized3", 0.8)])
@pytest.mark.parametrize("shape,steps,every", [((41, 65, 70), 7, 3), ((41, 65, 70), 40, 36), ((1, 40, 50), 7, 3)])
def test_states_agree(gpu_lib, storage, collision, tau, shape, steps, every):
    """Bit for bit those of steps one by one, at the end and after the reverse pass."""
    r1, r2, _ = wl.random_state(shape, seed=6, rho_lo=0.4, rho_hi=0.6, u_max=0.0)
    kw = dict(storage=storage, collision=collision, tau=(tau, tau), G12=-1.2)
    if storage.endswith("_dev"):
        kw["rho0_dev"] = 0.5
    lat = gpu_run(shape, r1, r2, None, 0, **kw)
    lat.record(steps, every)
    got = lat.get_populations()
    lat.adjoint(r1, r2)
    assert np.array_equal(got, lat.get_populations())
    lat.close()
    lat = gpu_run(shape, r1, r2, None, 0, **kw)
    for _ in range(steps):
        lat.step(1)
    assert np.array_equal(got, lat.get_populations())
    lat.close()

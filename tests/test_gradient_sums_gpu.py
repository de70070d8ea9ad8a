"""The initial-density gradient is summed in FP64, also where the reverse pass keeps one
sensitivity per component and cell (FP32, tau = 1)."""
import numpy as np
import pytest

from _helpers import gpu_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16_dev", "bf16_rel"])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("steps,every", [(1, 1), (6, 3), (7, 4), (25, 25)])
def test_more_than_24_bits(gpu_lib, storage, tau, masked, steps, every):
    """A sum of two FP32 values of unequal size that is rounded to FP32 has 24 bits
    everywhere; in FP64 it has more nearly everywhere.  And it is the FP64 pass's gradient to
    the roundings of the steps, 20 dependent ones each (16 bits: of the FP32 pass over
    states with one such rounding a step)."""
    shape = (12, 14, 40)
    state = wl.random_state(shape, seed=5, rho_lo=0.4, rho_hi=0.6, u_max=0.0)[:2]
    kw = dict(G12=-1.2, G21=-1.1, tau=(tau, tau))
    solid = None
    if masked:
        solid = (np.random.default_rng(2).random(shape) < 0.1).astype(np.uint8)
        kw["wall_model"] = "mirror"
    out = {}
    for st in (storage, "f64"):
        more = dict(rho0_dev=0.5) if st.endswith("_dev") else {}
        lat = gpu_run(shape, *state, None, 0, storage=st, solid=solid, **kw, **more)
        lat.record(steps, every)
        a, b, _ = lat.moments()
        d = np.empty(shape), np.empty(shape)
        lat.adjoint(2 * a, b - 0.3, *d)
        lat.close()
        out[st] = np.array(d)
    fluid = np.ones(shape, bool) if solid is None else solid == 0
    g, w = out[storage][:, fluid], out["f64"][:, fluid]
    assert (g.astype(np.float32) != g).mean() > 0.9
    eps = {"f32": 6.0e-8, "f16_dev": 2.0 ** -11, "bf16_rel": 2.0 ** -8}[storage]
    assert np.abs(g - w).max() < steps * 20 * eps * np.abs(w).max()

"""Steps captured into a caller's graph: every replay advances the state."""
import pytest

from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16_dev", "bf16_dev", "f16_rel", "f64"])
@pytest.mark.parametrize("collision,tau", [("bgk", 1.0), ("regularized", 0.8), ("regularized3", 0.8)])
@pytest.mark.parametrize("calls", [[4], [2], [3, 5], [2, 4]])
def test_replays_advance(gpu_lib, storage, collision, tau, calls):
    """Calls that sum to an even number of steps, replayed three times, against the same
    calls made three times, to the storage format's rounding of one step per step."""
    import torch
    from paper_1601_01237_gb300 import Lattice
    shape, vmax = (40, 65, 70), 0.7 / 3
    r1, r2, u = wl.random_state(shape, seed=4, rho_lo=0.3, rho_hi=0.7, u_max=0.02)
    kw = dict(storage=storage, collision=collision, tau=(tau, tau), G12=-1.2)
    if storage.endswith("_dev"):
        kw["rho0_dev"] = 0.5
    s = torch.cuda.Stream()
    state = []
    for captured in (True, False):
        lat = Lattice(shape, stream=s.cuda_stream, **kw)
        lat.step(2)                       # every kernel loaded before the capture
        lat.step(3)
        lat.init_fields(r1, r2, u)
        lat.sync()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                for n in calls:
                    lat.step(n)
            with torch.cuda.stream(s):
                for _ in range(3):
                    g.replay()
            lat.sync()
        else:
            for _ in range(3):
                for n in calls:
                    lat.step(n)
        state.append(lat.get_populations())
        lat.close()
    eps = {"f64": 2.0 ** -53, "f32": 2.0 ** -24, "f16_dev": 2.0 ** -11, "f16_rel": 2.0 ** -11}.get(storage, 2.0 ** -8)
    assert abs(state[0] - state[1]).max() < 3 * sum(calls) * 20 * eps * vmax

"""Centre of mass of the droplet statistics for origins outside the lattice."""
import numpy as np
import pytest

from _helpers import gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("origin", [(3.3, -4.7, 1e3), (np.inf, 2.0, 3.0), (1.0, -np.inf, 1e300), (31.7, 30.1, 29.3)])
def test_origin(gpu_lib, storage, origin):
    """One shift by a period where a coordinate lies more than half of one from the
    origin, then the mean; 1e-12 relative to the largest coordinate that is summed."""
    shape = (21, 40, 63)
    rng = np.random.default_rng(3)
    r1 = rng.uniform(0.2, 0.8, shape)
    lat = gpu_run(shape, r1, 1.0 - r1, None, 0, storage=storage, G12=-0.5)
    rho = lat.moments()[0]
    st = lat.droplet_stats(0.5, origin)
    lat.close()
    inside = rho > 0.5
    assert st["volume"] == inside.sum()
    ax = np.meshgrid(*[np.arange(n, dtype=np.float64) for n in shape], indexing="ij")[::-1]
    for d in range(3):
        n = shape[2 - d]
        r = ax[d][inside] - origin[d]
        r = np.where(r > 0.5 * n, r - n, np.where(r < -0.5 * n, r + n, r))
        want, got = r.mean(), st["com"][d]
        assert got == want if np.isinf(want) else abs(got - want) <= 1e-12 * np.abs(r).max()

"""Rounding of the collision: nothing that all directions of a cell share may leave a
trace in the mass, and the parameter derivatives of long runs carry no more of it than
an FP32 value of their size."""
import numpy as np
import pytest

from _helpers import gpu_run
from paper_1601_01237_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("collision,tau,forcing", [("bgk", 1.0, "edm"), ("bgk", 0.8, "edm"), ("bgk", 0.8, "guo"),
                                                   ("regularized", 0.8, "edm"), ("regularized3", 0.8, "guo")])
@pytest.mark.parametrize("storage,eps", [("f64", 2.0 ** -53), ("f32", 2.0 ** -24)])
def test_mass_of_one_step_has_no_bias(gpu_lib, storage, eps, collision, tau, forcing):
    """Mean relative change of mass over 64^3 cells of two components: a cell's change
    is below 2 roundings rms (its density is a sum of 19 terms), so that the mean stays
    within 5 standard errors, 10 eps / sqrt(2 N).  From the second step on: the 19 products
    of one density that a state starts from are not a collision's output."""
    shape = (64, 64, 64)
    r1, r2, u = wl.random_state(shape, seed=21, rho_lo=0.2, rho_hi=0.9, u_max=0.05)
    lat = gpu_run(shape, r1, r2, u, 0, storage=storage, collision=collision, tau=(tau, tau), forcing=forcing, G12=-0.6)
    lat.step(1)
    mass = []
    for _ in range(2):
        mass.append(np.sum(lat.get_populations().astype(np.longdouble)))
        lat.step(1)
    lat.close()
    assert abs(float((mass[1] - mass[0]) / mass[0])) < 10 * eps / np.sqrt(2.0 * np.prod(shape))


def test_parameter_derivatives(gpu_lib):
    """dL/dG12, dL/dG21, dL/dtau1 and dL/dtau2 of an FP32 droplet run, each against its
    own FP64 value.  Each is a sum of terms of both signs, so that its rounding does not
    shrink where the sum does: over six starts, half a unit in the last place of the
    largest value it takes."""
    n, steps = 96, 50
    z, y, x = np.meshgrid(*[np.arange(n, dtype=np.float64)] * 3, indexing="ij")
    c = (n - 1) / 2
    q = np.sqrt(((z - c) / (0.17 * n)) ** 2 + ((y - c) / (0.21 * n)) ** 2 + ((x - c) / (0.25 * n)) ** 2)
    target = 0.03 + 0.485 * (1.0 - np.tanh(0.1 * n * (q - 1.0)))
    rng = np.random.default_rng(8)
    par = []
    for _ in range(6):
        cen, R = (n - 1) * rng.uniform(0.45, 0.55, 3), n * rng.uniform(0.2, 0.25)
        dist = np.sqrt((z - cen[0]) ** 2 + (y - cen[1]) ** 2 + (x - cen[2]) ** 2)
        a = (0.148 + 0.3745 * (1.0 - np.tanh((dist - R) / 2.0))) * (1.0 + 1e-3 * rng.uniform(-1, 1, dist.shape))
        b = 1.045 - a
        for storage in ("f32", "f64"):
            lat = gpu_run(a.shape, a, b, None, 0, storage=storage, G12=-1.8)
            lat.record(steps, 25)
            f1, f2, _ = lat.moments()
            par.append(lat.adjoint(2 * (f1 - target) + 0.5 * f2, 0.5 * f1))
            lat.close()
    f32, f64 = np.array(par[0::2]), np.array(par[1::2])
    off = np.abs(f32 - f64).max(0) / np.abs(f64).max(0)
    assert (off < 2.0 ** -24).all(), off


@pytest.mark.parametrize("collision,tau", [("bgk", 1.0), ("regularized", 0.7)])
def test_runs_round_no_more_along_z(gpu_lib, collision, tau):
    """A run of steps in one call marches along z and collects a cell's momentum and
    density gradient in z from planes that come one after another: its velocity errors
    are no larger, along every axis, than those of the same steps made one by one, which
    subtract opposite populations and neighbours first."""
    import torch
    from paper_1601_01237_gb300 import Lattice
    shape, steps = (64, 64, 64), 20
    err = np.zeros((2, 3))
    for seed in (1, 2):
        rng = np.random.default_rng(seed)
        r1, r2 = [torch.from_numpy(0.5 * (1.0 + 0.01 * rng.uniform(-1, 1, shape))).cuda() for _ in range(2)]
        u = []
        for storage, calls in (("f64", [steps]), ("f32", [1] * steps), ("f32", [steps])):
            lat = Lattice(shape, storage=storage, G12=-1.2, collision=collision, tau=(tau, tau))
            lat.init_fields(r1, r2)
            for n in calls:
                lat.step(n)
            u.append(torch.zeros(shape + (3,), dtype=torch.float64, device="cuda"))
            lat.moments_device(None, None, u[-1], out_f64=True)
            lat.close()
        for k in (0, 1):
            err[k] += (u[k + 1] - u[0]).square().mean(dim=(0, 1, 2)).cpu().numpy()
    assert (err[1] <= err[0]).all(), np.sqrt(err[1] / err[0])

"""Sites without an ordinary density: u = (j + F/2)/rho keeps the value of a
division where the reciprocal form has none. Density zero gives signed
infinities, a density beyond the doubles gives zero, and such a velocity
enters the FP64 collisions as it stands."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import inputs, ld  # noqa: E402

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
SITE = (1, 3, 5)  # z, y, x
MODEL = dict(tau_f=0.8, tau_g=1.3, kappa=0.05)


def distributions(nx, ny, nz):
    f = np.broadcast_to(W[:, None, None, None], (19, nz, ny, nx)).copy()
    g = W[:, None, None, None] * inputs.spinodal_phi(nx, ny, nz, seed=3, amplitude=0.5)
    return f, g


def site(a):
    return a.cpu().numpy()[(..., *SITE)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("force", ["potential", "stress"])
def test_moments(precision, stencil, force):
    nx, ny, nz = 11, 6, 5
    sim = ld.LdSim(nx, ny, nz, precision=precision, stencil=stencil, force=force, **MODEL)
    f, g = distributions(nx, ny, nz)

    def u_with(values):
        state = f.copy()
        state[(slice(None), *SITE)] = values
        sim.set_distributions(torch.from_numpy(state), torch.from_numpy(g))
        return site(sim.moments()["u"])

    half_force = u_with(W)  # density 1, no momentum but rounding's
    assert (np.abs(half_force) > 1e-6).all()
    assert np.array_equal(u_with(0.0 * W), np.copysign(np.inf, half_force))
    rest = 0.0 * W
    rest[0] = np.inf  # j sums c_i f_i: 0 x inf leaves it undefined
    assert np.isnan(u_with(rest)).all()
    if precision == "fp64":  # the density overflows, j does not
        assert (u_with(np.full(19, 1.5e307)) == 0.0).all()


@pytest.mark.parametrize("kernel,collision", [("generic", "bgk"), ("generic", "trt"), ("fused", "bgk")])
def test_fp64_step_with_infinite_density(kernel, collision):
    """u = j/inf = 0: the site's g relaxes to the equilibrium at rest, and only f is lost."""
    nx, ny, nz = 32, 8, 4
    sim = ld.LdSim(nx, ny, nz, precision="fp64", kernel=kernel, collision=collision, **MODEL)
    f, g = distributions(nx, ny, nz)
    f[(0, *SITE)] = np.inf
    sim.set_distributions(torch.from_numpy(f), torch.from_numpy(g))
    sim.step(1)
    got_f, got_g = (t.cpu().numpy() for t in sim.distributions())
    phi = g.sum(axis=0)
    lap = sum(np.roll(phi, d, a) for a in range(3) for d in (1, -1)) - 6 * phi
    p = phi[SITE]
    mu = -0.0625 * p + 0.0625 * p ** 3 - MODEL["kappa"] * lap[SITE]
    dev = 0.5 * mu - p / 3
    for i in range(19):
        z, y, x = ((SITE[a] + C[i][2 - a]) % n for a, n in enumerate((nz, ny, nx)))
        geq = W[i] * (p + 4.5 * dev * ((C[i] ** 2).sum() - 1))
        old = g[(i, *SITE)]
        assert abs(got_g[i, z, y, x] - (old - (old - geq) / MODEL["tau_g"])) <= 1e-15
        assert not np.isfinite(got_f[i, z, y, x])
    assert np.isfinite(got_g).all()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_crystal_velocity_at_zero_density(precision):
    nx, ny, nz = 11, 6, 5
    rng = np.random.default_rng(2)
    q = torch.from_numpy(0.2 * rng.standard_normal((5, nz, ny, nx)))
    sim = ld.LcSim(nx, ny, nz, precision=precision)
    rho = np.ones((nz, ny, nx))
    sim.init(q, torch.from_numpy(rho))
    half_force = site(sim.fields()["u"])
    rho[SITE] = 0.0
    sim.init(q, torch.from_numpy(rho))
    u = site(sim.fields()["u"])
    assert (np.abs(half_force) > 1e-6).all()
    assert np.array_equal(u, np.copysign(np.inf, half_force))  # FP32: the reciprocal of zero is infinite too

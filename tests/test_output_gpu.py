"""Initial state and macroscopic output on the GPU where their FP32-pipe forms
could go wrong: rounding of the 16-bit initial deviations, the moments' error-
free float sums and integer conversions at extreme values, lattices whose
size is not a multiple of the vectors that the totals load."""

import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import inputs, ld  # noqa: E402

pytestmark = pytest.mark.gpu

STORE = {"fp32": torch.float32, "fp16dev": torch.float16, "bf16dev": torch.bfloat16, "fp64": torch.float64}


def planes(sim, precision):
    nz, ny, nx = sim.shape
    out = torch.empty((38, nz, ny, nx), dtype=STORE[precision], device="cuda")
    ld.ld_pack_planes(sim.ctx, 0, nz, out)
    return out


def round_once(x, bits, emin):
    """float64 x rounded to nearest even with `bits` significant bits and least exponent emin."""
    _, e = np.frexp(x)
    step = np.ldexp(1.0, np.maximum(e - bits, emin - bits + 1))
    return np.rint(x / step) * step


@pytest.mark.parametrize("precision,bits,emin", [("fp16dev", 11, -14), ("bf16dev", 8, -126)])
def test_initial_deviations_are_rounded_once(precision, bits, emin):
    """At rest f_i = w_i rho, one FP32 product. With rho away from rho0 = 1 the FP32 difference to the
    reference is inexact, and rounding it again would differ from rounding the exact one."""
    nx, ny, nz = 40, 12, 9
    phi = np.zeros((nz, ny, nx))
    rho = np.random.default_rng(4).uniform(0.1, 8.0, phi.shape)
    sim = ld.LdSim(nx, ny, nz, precision=precision)
    sim.init(torch.from_numpy(phi).cuda(), torch.from_numpy(rho).cuda())
    got = planes(sim, precision)[:19].double().cpu().numpy()
    w = np.array([np.float32(1) / np.float32(3)] + [np.float32(1) / np.float32(18)] * 6
                 + [np.float32(1) / np.float32(36)] * 12, np.float32)[:, None, None, None]
    ref = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12).astype(np.float32)[:, None, None, None]
    exact = (w * rho.astype(np.float32)).astype(np.float64) - ref.astype(np.float64)
    once = round_once(exact, bits, emin)
    assert np.array_equal(got, once)
    twice = round_once(exact.astype(np.float32).astype(np.float64), bits, emin)
    assert precision == "bf16dev" or (twice != once).any()


@pytest.mark.parametrize("case", ["ordinary", "wide", "subnormal", "huge", "inf", "nan", "zero"])
@pytest.mark.parametrize("stencil", [7, 19])
def test_moments_of_extreme_states(case, stencil):
    nx, ny, nz = 11, 6, 5
    rng = np.random.default_rng(5)
    f = rng.random((19, nz, ny, nx)) * 0.1 + 0.01
    g = rng.standard_normal((19, nz, ny, nx)) * 0.1
    if case == "wide":  # values spanning more bits than a double holds
        g *= np.float64(2.0) ** rng.integers(-70, 5, g.shape)
    elif case == "subnormal":
        g *= 2.0 ** -130
    elif case == "huge":  # the float sum overflows, the double one does not
        f[:, 1, 2, 3] = 3.0e38
    elif case == "inf":
        f[4, 1, 2, 3] = math.inf
        g[7, 2, 1, 0] = -math.inf
    elif case == "nan":
        f[4, 1, 2, 3] = math.nan
    elif case == "zero":
        g[:] = 0.0
    f, g = (a.astype(np.float32).astype(np.float64) for a in (f, g))  # what the state holds
    sim = ld.LdSim(nx, ny, nz, precision="fp32", stencil=stencil)
    sim.set_distributions(torch.from_numpy(f), torch.from_numpy(g))
    m = {k: v.cpu().numpy() for k, v in sim.moments(grad_phi=True).items()}
    exact = lambda a: np.array([math.fsum(v) if np.isfinite(v).all() else v.sum()  # noqa: E731
                                for v in a.reshape(19, -1).T]).reshape(a.shape[1:])
    # a sum of 19 doubles is within 18 units of 2^-53 of the sum of magnitudes
    for key, a in (("rho", f), ("phi", g)):
        want, tol = exact(a), 18 * 2.0 ** -53 * np.abs(a).sum(axis=0)
        fine = np.isfinite(want)
        assert np.array_equal(np.isnan(m[key]), np.isnan(want))
        assert np.array_equal(m[key][~fine & ~np.isnan(want)], want[~fine & ~np.isnan(want)])
        assert (np.abs(m[key] - want)[fine] <= tol[fine]).all()
    if case in ("ordinary", "wide", "zero"):  # u = (j + F/2)/rho with F = -phi grad(mu) of the FP32 mu
        assert np.isfinite(m["u"]).all() and np.isfinite(m["grad_phi"]).all()
        phi32 = np.zeros(g.shape[1:], np.float32)
        for i in range(19):
            phi32 = phi32 + g[i].astype(np.float32)
        roll = lambda h, a, d: np.roll(h, -d, axis=2 - a)  # noqa: E731
        p = phi32.astype(np.float64)
        if stencil == 7:
            want = np.stack([0.5 * (roll(p, a, 1) - roll(p, a, -1)) for a in range(3)])
            assert np.abs(m["grad_phi"] - want).max() <= 2.0 ** -53 * np.abs(p).max()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("dims", [(5, 5, 5), (33, 7, 5), (64, 8, 4), (31, 30, 29)])
def test_totals_of_sizes_off_the_vectors(precision, dims):
    nx, ny, nz = dims
    sim = ld.LdSim(nx, ny, nz, precision=precision)
    sim.workspace.fill_(255)  # NaN in the padding of every row, which must not be added
    sim.close()
    sim.ctx = ld.ld_create(nx, ny, nz, sim.params, sim.workspace)
    sim.init(torch.from_numpy(inputs.spinodal_phi(nx, ny, nz, seed=6, amplitude=0.4)).cuda())
    f, g = (t.cpu().numpy() for t in sim.distributions())
    got = sim.totals().cpu().numpy()
    n = nx * ny * nz
    # each site's 19 values are summed in the arithmetic type: at most 18 roundings of the sum of magnitudes
    unit = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    want = np.array([f.sum(), g.sum()])
    tol = 20 * unit * np.array([np.abs(f).sum(), np.abs(g).sum()]) + n * 2.0 ** -52
    assert (np.abs(got[:2] - want) <= tol).all()
    assert np.abs(got[2:]).max() <= 20 * unit * np.abs(f).sum()


@pytest.mark.parametrize("precision", ["fp16dev", "bf16dev"])
def test_initial_zeros_keep_their_sign(precision):
    """phi = +-2^-149 with mean 0: the references are 0 and w_i phi along the axes underflows to a zero with phi's
    sign, which the deviation of the FP64 form, x - 0, keeps."""
    nx, ny, nz = 10, 6, 5
    phi = np.full(nx * ny * nz, 2.0 ** -149)
    phi[1::2] *= -1.0
    phi = phi.reshape(nz, ny, nx)
    sim = ld.LdSim(nx, ny, nz, precision=precision)
    sim.init(torch.from_numpy(phi))
    bits = planes(sim, precision)[20:26].view(torch.int16).cpu().numpy().view(np.uint16)
    assert np.array_equal(bits, np.broadcast_to(np.where(phi < 0, 0x8000, 0).astype(np.uint16), bits.shape))


def fma32(a, b, c):
    """float32 a b + c with one rounding: the exact product's float64 sum rounded to odd, then to float32."""
    p, c = a.astype(np.float64) * b, np.asarray(c, np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    odd = (s.view(np.int64) & 1).astype(bool)
    s = np.where((err != 0) & ~odd, np.nextafter(s, np.copysign(np.inf, err)), s)
    return s.astype(np.float32)


C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def f32(v, like):
    return np.full_like(like, np.float32(v))


def dot(c, u):
    cu = np.zeros_like(u[0])
    for k, v in zip(c, u):
        cu = cu + v if k > 0 else cu - v if k < 0 else cu
    return cu


def feq32(i, rho, u, uu):
    cu = dot(C[i], u)
    w = np.float32(1) / np.float32(3 if i == 0 else 18 if i <= 6 else 36)
    return (w * rho) * fma32(f32(-1.5, uu), uu, fma32(np.float32(4.5) * cu, cu, fma32(f32(3, cu), cu, f32(1, cu))))


@pytest.mark.parametrize("stencil", [7, 19])
def test_fp32_initial_state_has_the_written_fusions(stencil):
    """Bit for bit feq and geq with one rounding where the code says so, mu of phi included."""
    nx, ny, nz = 13, 7, 6
    rng = np.random.default_rng(12)
    phi, rho = 0.4 * rng.standard_normal((nz, ny, nx)), 1.0 + 0.05 * rng.standard_normal((nz, ny, nx))
    u = 0.05 * rng.standard_normal((3, nz, ny, nx))
    prm = dict(A=-0.07, B=0.051, kappa=0.043, Gamma=0.37)
    sim = ld.LdSim(nx, ny, nz, precision="fp32", stencil=stencil, **prm)
    sim.init(*(torch.from_numpy(a) for a in (phi, rho, u)))
    got = planes(sim, "fp32").cpu().numpy()
    A, B, kappa, Gamma = (np.float32(prm[k]) for k in ("A", "B", "kappa", "Gamma"))
    p, rho, u = phi.astype(np.float32), rho.astype(np.float32), u.astype(np.float32)
    at = lambda c: np.roll(p, (-c[2], -c[1], -c[0]), (0, 1, 2))  # noqa: E731
    if stencil == 7:
        lap = at(C[1])
        for i in range(2, 7):
            lap = lap + at(C[i])
        lap = fma32(f32(-6, p), p, lap)
    else:
        lap = np.zeros_like(p)
        for i in range(1, 19):
            lap = fma32(np.float32(1) / f32(3 if i <= 6 else 6, p), at(C[i]) - p, lap)
    mu = fma32(f32(-kappa, p), lap, fma32(f32(A, p), p, B * p * p * p))
    uu = fma32(u[2], u[2], fma32(u[0], u[0], u[1] * u[1]))
    dev45 = np.float32(4.5) * fma32(f32(Gamma, p), mu, -(p / np.float32(3)))
    for i in range(19):
        cu, w = dot(C[i], u), np.float32(1) / np.float32(3 if i == 0 else 18 if i <= 6 else 36)
        t = fma32(np.float32(3) * p, cu, p)
        t = t + dev45 if i > 6 else t - dev45 if i == 0 else t
        t = fma32(-(np.float32(1.5) * p), uu, fma32((np.float32(4.5) * p) * cu, cu, t))
        assert np.array_equal(got[i], feq32(i, rho, u, uu)) and np.array_equal(got[19 + i], w * t)


def test_fp32_crystal_initial_state_has_the_written_fusions():
    nx, ny, nz = 13, 7, 6
    rng = np.random.default_rng(13)
    q, rho = 0.2 * rng.standard_normal((5, nz, ny, nx)), 1.0 + 0.05 * rng.standard_normal((nz, ny, nx))
    u = 0.05 * rng.standard_normal((3, nz, ny, nx))
    sim = ld.LcSim(nx, ny, nz, precision="fp32")
    sim.init(*(torch.from_numpy(a) for a in (q, rho, u)))
    got = sim.fields()["f"].cpu().numpy()
    rho, u = rho.astype(np.float32), u.astype(np.float32)
    uu = fma32(u[2], u[2], fma32(u[1], u[1], u[0] * u[0]))
    for i in range(19):
        assert np.array_equal(got[i], feq32(i, rho, u, uu).astype(np.float64))


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("force", ["potential", "stress"])
def test_velocity_and_gradient_values(precision, stencil, force, orc):
    """u = (j + F/2)/rho and grad phi in FP64 from the state's values, F from the phi, mu and P that the arithmetic
    of the precision gives: phi and mu of the FP32 forms bit for bit, P to its rounding."""
    nx, ny, nz = 11, 6, 5
    rng = np.random.default_rng(21)
    phi0, rho0 = 0.4 * rng.standard_normal((nz, ny, nx)), 1.0 + 0.05 * rng.standard_normal((nz, ny, nx))
    u0 = 0.05 * rng.standard_normal((3, nz, ny, nx))
    A, B, kappa = -0.07, 0.051, 0.043
    sim = ld.LdSim(nx, ny, nz, precision=precision, stencil=stencil, force=force, A=A, B=B, kappa=kappa, tau_f=0.8)
    sim.init(*(torch.from_numpy(a) for a in (phi0, rho0, u0)))
    sim.step(2)
    m = {k: v.cpu().numpy() for k, v in sim.moments(grad_phi=True).items()}
    f, g = (t.cpu().numpy() for t in sim.distributions())  # FP32 values, or reference + deviation, exact in FP64
    real = np.float64 if precision == "fp64" else np.float32
    unit = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    phi = np.zeros((nz, ny, nx), real)
    for i in range(19):
        phi = phi + g[i].astype(real)
    if stencil == 7:
        lap = sum((np.roll(phi, s, a) for a in (2, 1, 0) for s in (-1, 1)), real(0)) - real(6) * phi
    else:
        lap = np.zeros_like(phi)
        for i in range(1, 19):
            lap = lap + real(1) / real(3 if i <= 6 else 6) * (np.roll(phi, (-C[i][2], -C[i][1], -C[i][0]), (0, 1, 2)) - phi)
    mu = (real(A) * phi + real(B) * phi * phi * phi) - real(kappa) * lap
    phi, mu = phi.astype(np.float64), mu.astype(np.float64)
    exact = lambda a: np.array([math.fsum(v) for v in a.reshape(19, -1).T]).reshape(a.shape[1:])  # noqa: E731
    c = np.array(C, float)
    j = np.stack([exact(c[:, a, None, None, None] * f) for a in range(3)])
    size = np.abs(f).sum(axis=0)
    if force == "potential":
        F = -exact(g) * orc.gradient(mu, stencil)
        # FP32: the same mu; FP64: its own to a few units of its terms, over a gradient of weight 1
        mu_terms = np.abs(A * phi).max() + np.abs(B * phi ** 3).max() + kappa * 12 * np.abs(phi).max()
        f_err = 2.0 ** -53 * 64 * np.abs(phi).max() * mu_terms
    else:
        prm = orc.param_vector(A=float(real(A)), B=float(real(B)), kappa=float(real(kappa)), stencil=stencil, force="stress")
        P = orc.stress(phi, prm)
        F = -np.stack([sum(orc.gradient(P[k], stencil)[b] for b, k in enumerate(ks))
                       for ks in ((0, 3, 4), (3, 1, 5), (4, 5, 2))])
        # about 40 roundings of the terms of P (phi lap phi the largest), and three gradients of it
        f_err = unit * 3 * 40 * (np.abs(P).max() + kappa * 12 * np.abs(phi).max() ** 2)
    rho = exact(f)
    tol = (2.0 ** -53 * 24 * (size + np.abs(F).max()) + f_err) / rho
    assert np.abs(F).max() > 1e3 * f_err  # the force is there to be seen
    assert (np.abs(m["u"] - (j + 0.5 * F) / rho) <= tol).all()
    phi_err = 0.0 if precision != "fp64" else 18 * 2.0 ** -53 * np.abs(g).sum(axis=0).max()
    assert np.abs(m["grad_phi"] - orc.gradient(phi, stencil)).max() <= 16 * 2.0 ** -53 * np.abs(phi).max() + phi_err

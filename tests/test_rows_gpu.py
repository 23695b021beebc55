"""The site-ordered launches (LD_KERNEL_GENERIC): mu formed in the collision from
phi equals the mu launch's, blocks across the ends of rows, state and fields
buffers that are aligned to single values only."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import inputs, ld  # noqa: E402

pytestmark = pytest.mark.gpu

MODEL = dict(tau_f=0.8, tau_g=1.3, kappa=0.05)


def started(nx, ny, nz, **kw):
    sim = ld.LdSim(nx, ny, nz, kernel="generic", **MODEL, **kw)
    rng = np.random.default_rng(nx + ny + nz)
    phi = inputs.spinodal_phi(nx, ny, nz, seed=8, amplitude=0.5)
    sim.init(*(torch.from_numpy(a).cuda() for a in (phi, 1.0 + 0.02 * rng.standard_normal(phi.shape),
                                                    0.02 * rng.standard_normal((3, *phi.shape)))))
    return sim


@pytest.mark.parametrize("dims", [(4, 4, 4), (5, 4, 6), (127, 5, 4), (128, 4, 5), (129, 6, 4), (33, 31, 7)])
@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "bf16dev"])
def test_fields_of_a_step_are_mu_of_its_phi(dims, precision):
    nx, ny, nz = dims
    n, npad = nx * ny * nz, -(-nx * ny * nz // 64) * 64
    sim = started(nx, ny, nz, precision=precision)
    sim.step(2)
    src, dst = sim.save_state(), torch.empty(ld.ld_state_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
    fld = torch.zeros(ld.ld_fields_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
    ld.ld_step_between(sim.ctx, src, dst, fld)
    phi, mu = (a[:n].view(nz, ny, nx).cpu().numpy() for a in fld.view(torch.float32)[:2 * npad].view(2, npad))
    nb = np.zeros_like(phi)
    for axis in (2, 1, 0):  # the kernels' order: +x, -x, +y, -y, +z, -z, each addition rounded to float
        nb = nb + np.roll(phi, -1, axis) if axis < 2 else np.roll(phi, -1, axis)
        nb = nb + np.roll(phi, 1, axis)
    A, B, kappa = (np.float32(v) for v in (-0.0625, 0.0625, 0.05))
    lap = nb - np.float32(6) * phi
    want = (A * phi + B * phi * phi * phi) - kappa * lap
    assert np.array_equal(mu, want)
    # and the step that used them is the one from the same state in the context
    sim.step(1)
    after = sim.save_state()
    nbytes = 38 * npad * (4 if precision == "fp32" else 2)
    pad = torch.arange(nbytes // (nbytes // (38 * npad)), device="cuda") % npad < n
    a, b = (t[:nbytes].view(38 * npad, -1)[pad] for t in (after, dst))
    assert torch.equal(a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp16dev"])
def test_adjoint_step_from_an_unaligned_state(precision):
    nx, ny, nz = 9, 7, 6
    sim = started(nx, ny, nz, precision=precision)
    work = torch.empty(ld.ld_adjoint_workspace_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
    ld.ld_adjoint_attach(sim.ctx, work)
    seed = torch.rand((nz, ny, nx), dtype=torch.float64, device="cuda")
    state = sim.save_state()
    step = 4 if precision == "fp32" else 2
    moved = torch.empty(state.numel() + step, dtype=torch.uint8, device="cuda")[step:]
    moved.copy_(state)
    out = []
    for s in (state, moved):
        grad = torch.zeros(2, dtype=torch.float64, device="cuda")
        ld.ld_adjoint_seed(sim.ctx, seed)
        ld.ld_adjoint_step(sim.ctx, s, grad)
        f = torch.empty((19, nz, ny, nx), dtype=torch.float64, device="cuda")
        g = torch.empty_like(f)
        ld.ld_adjoint_get(sim.ctx, f, g)
        out.append((f, g, grad))
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("dims", [(4, 4, 4), (5, 4, 7), (33, 9, 5), (129, 6, 4)])
@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("collision", ["bgk", "trt"])
@pytest.mark.parametrize("stencil", [7, 19])
def test_one_step_with_the_stress_force(dims, precision, collision, stencil, orc):
    """One step with F = -div P from a stored state in flow, against the oracle's from the same state, and the
    fields it leaves: formed in the collision (7-point) and from the stress launch (19-point). Dimensions of 4 and 5, where +2 and -2 meet or wrap, and blocks across the ends of rows."""
    nx, ny, nz = dims
    n, npad = nx * ny * nz, -(-nx * ny * nz // 64) * 64
    sim = started(nx, ny, nz, precision=precision, force="stress", collision=collision, stencil=stencil)
    phi0 = inputs.spinodal_phi(nx, ny, nz, seed=8, amplitude=0.5)
    sim.step(2)
    f0, g0 = (t.cpu().numpy() for t in sim.distributions())
    src = sim.save_state()
    dst = src.clone()  # with the references, which the step does not write
    fld = torch.zeros(ld.ld_fields_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
    ld.ld_step_between(sim.ctx, src, dst, fld)
    sim.load_state(dst)
    got = np.concatenate([t.cpu().numpy() for t in sim.distributions()])
    phi, mu = (a[:n].view(nz, ny, nx).cpu().numpy() for a in fld.view(torch.float32)[:2 * npad].view(2, npad))
    # phi: 18 roundings of the magnitudes (19 more where the values are decoded); mu: the operations of the mu launch
    assert (np.abs(phi - g0.sum(axis=0)) <= 38 * 2.0 ** -24 * np.abs(g0).sum(axis=0)).all()
    c, w = orc.lattice()
    one = np.float32(1)
    if stencil == 7:
        nb = np.zeros_like(phi)
        for axis in (2, 1, 0):
            nb = nb + np.roll(phi, -1, axis) if axis < 2 else np.roll(phi, -1, axis)
            nb = nb + np.roll(phi, 1, axis)
        lap = nb - np.float32(6) * phi
    else:
        lap = np.zeros_like(phi)
        for i in range(1, 19):
            lap = lap + one / np.float32(3 if i <= 6 else 6) * (np.roll(phi, -c[i][::-1], (0, 1, 2)) - phi)
    A, B, kappa = (np.float32(v) for v in (-0.0625, 0.0625, 0.05))
    assert np.array_equal(mu, (A * phi + B * phi * phi * phi) - kappa * lap)
    prm = orc.param_vector(**dict(MODEL, kappa=float(kappa)), force="stress", collision=collision, stencil=stencil)
    want = np.concatenate(orc.step(f0, g0, prm))
    # FP32: about 60 operations reach a population, on terms no larger than the density
    tol = 64 * 2.0 ** -24 * f0.sum(axis=0).max()
    if precision != "fp32":  # and half a unit of the stored deviation
        pb = phi0.mean()
        dev = 0.5 * (-0.0625 * pb + 0.0625 * pb ** 3) - pb / 3
        ref = np.concatenate([w, w * (pb + 4.5 * dev * ((c ** 2).sum(axis=1) - 1))])[:, None, None, None]
        half = 2.0 ** -11 if precision == "fp16dev" else 2.0 ** -8
        tol = tol * (1 + half) + half * np.abs(want - ref) + 2.0 ** -24
    assert (np.abs(got - want) <= tol).all()

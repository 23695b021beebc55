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

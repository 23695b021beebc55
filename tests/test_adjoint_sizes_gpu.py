"""The adjoint's launches by lattice size: two periods of a lattice along z, on
the other side of the line where k_adj_mu takes four sites a thread, have the
same adjoint at every site and twice the parameters' gradients."""

import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import inputs, ld  # noqa: E402

pytestmark = pytest.mark.gpu


def reverse_step(phi, seed, precision, stencil):
    nz, ny, nx = phi.shape
    sim = ld.LdSim(nx, ny, nz, precision=precision, stencil=stencil, tau_f=0.8, tau_g=1.3, kappa=0.05)
    sim.init(phi)
    sim.step(2)
    work = torch.empty(ld.ld_adjoint_workspace_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
    ld.ld_adjoint_attach(sim.ctx, work)
    grad = torch.zeros(2, dtype=torch.float64, device="cuda")
    ld.ld_adjoint_seed(sim.ctx, seed)
    for _ in range(2):
        ld.ld_adjoint_step(sim.ctx, sim.save_state(), grad)
    f = torch.empty((19, nz, ny, nx), dtype=torch.float64, device="cuda")
    g = torch.empty_like(f)
    ld.ld_adjoint_get(sim.ctx, f, g)
    return f, g, grad


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("stencil", [7, 19])
@pytest.mark.parametrize("dims", [(70, 68, 33), (67, 61, 39)])
def test_two_periods_have_twice_the_gradient(precision, stencil, dims):
    nx, ny, nz = dims  # 157,080 and 159,393 sites, below 1216 blocks of 256; two periods are above
    phi = torch.from_numpy(inputs.spinodal_phi(nx, ny, nz, seed=3, amplitude=0.4)).cuda()
    seed = torch.rand((nz, ny, nx), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    f, g, grad = reverse_step(phi, seed, precision, stencil)
    f2, g2, grad2 = reverse_step(torch.cat([phi, phi]), torch.cat([seed, seed]), precision, stencil)
    assert torch.equal(f2[:, :nz], f) and torch.equal(f2[:, nz:], f)
    assert torch.equal(g2[:, :nz], g) and torch.equal(g2[:, nz:], g)
    # FP64 sums of the same terms in another order
    assert ((grad2 - 2 * grad).abs() <= 1e-9 * grad.abs()).all() and (grad != 0).all()

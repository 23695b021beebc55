"""The one-launch step of small lattices (LD_KERNEL_AUTO) gives the bits of the
kernel that AUTO takes for larger lattices: fused where the lattice is tiled,
else generic. Tiles that reach past the lattice, halos that wrap more than
once, every option, consecutive launches that overlap, the fields output,
streams and capture."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import inputs, ld  # noqa: E402

pytestmark = pytest.mark.gpu

DIMS = [(4, 4, 4), (5, 4, 7), (31, 5, 6), (32, 4, 4), (32, 8, 4), (33, 9, 5), (64, 8, 4), (70, 6, 10), (24, 50, 40),
        (32, 40, 48)]
MODEL = dict(tau_f=0.8, tau_g=1.3, kappa=0.05)


def fields(nx, ny, nz):
    rng = np.random.default_rng(nx * ny + nz)
    phi = inputs.spinodal_phi(nx, ny, nz, seed=9, amplitude=0.5)
    rho = 1.0 + 0.02 * rng.standard_normal(phi.shape)
    u = 0.02 * rng.standard_normal((3, *phi.shape))
    return [torch.from_numpy(a).cuda() for a in (phi, rho, u)]


def pair(nx, ny, nz, **model):
    other = "fused" if nx % 32 == 0 and ny % 8 == 0 and nz % 4 == 0 else "generic"
    sims = [ld.LdSim(nx, ny, nz, kernel=k, **MODEL, **model) for k in ("auto", other)]
    assert ld.ld_step_kernel(sims[0].ctx) == other
    start = fields(nx, ny, nz)
    for sim in sims:
        sim.init(*start)
    return sims


def planes(sim):
    out = torch.empty((38, *sim.shape), dtype=torch.float32, device="cuda")
    ld.ld_pack_planes(sim.ctx, 0, sim.nz, out)
    return out


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("stencil", [7, 19])
def test_bits_do_not_depend_on_the_kernel(dims, stencil):
    small, other = pair(*dims, stencil=stencil)
    for steps in (1, 6):
        small.step(steps)
        other.step(steps)
        assert torch.equal(planes(small), planes(other))
    small.check()


def test_fields_output_and_state_between_buffers():
    nx, ny, nz = 37, 10, 6
    n, npad = nx * ny * nz, -(-nx * ny * nz // 64) * 64
    got = []
    for sim in pair(nx, ny, nz):
        src, dst = sim.save_state(), torch.zeros(ld.ld_state_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
        fld = torch.zeros(ld.ld_fields_bytes(sim.ctx), dtype=torch.uint8, device="cuda")
        ld.ld_step_between(sim.ctx, src, dst, fld)
        sim.load_state(dst)
        got.append((fld.view(torch.float32)[:2 * npad].view(2, npad)[:, :n], planes(sim)))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


def test_overlapping_launches_on_a_stream_and_in_a_graph():
    small, other = pair(32, 24, 20)
    checkpoint = small.save_state()
    other.step(40)
    want = planes(other)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    ld.ld_set_stream(small.ctx, stream.cuda_stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        small.step(10)  # an even number: the state returns to its first buffer
    with torch.cuda.stream(stream):
        small.load_state(checkpoint)
        for _ in range(4):
            graph.replay()
        got = planes(small)
    stream.synchronize()
    assert torch.equal(got, want)

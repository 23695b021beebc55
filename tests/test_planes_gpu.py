"""ld_pack_planes / ld_unpack_planes over every copy width: plane sizes and
buffers that are aligned to 16, 8, 4 and 2 bytes only, wrapping ranges, and the
whole lattice with and without padding."""

import pytest

torch = pytest.importorskip("torch")

from paper_1609_01479_gb300 import ld  # noqa: E402

pytestmark = pytest.mark.gpu

STORE = {"fp64": torch.float64, "fp32": torch.float32, "fp16dev": torch.float16}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16dev"])
@pytest.mark.parametrize("dims", [(32, 8, 4), (5, 5, 5), (6, 5, 7), (4, 4, 9), (64, 30, 11)])
@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_planes_survive_the_round_trip(precision, dims, offset):
    nx, ny, nz = dims
    sim = ld.LdSim(nx, ny, nz, precision=precision)
    f = torch.rand((19, nz, ny, nx), dtype=torch.float64, device="cuda")
    g = torch.rand((19, nz, ny, nx), dtype=torch.float64, device="cuda")
    sim.set_distributions(f, g)
    state = torch.cat(sim.distributions())
    for z0, count in ((0, nz), (1, 2), (nz - 1, 3), (-2, nz), (2, 1)):
        buf = torch.full((38 * count * ny * nx + offset,), 7.0, dtype=STORE[precision], device="cuda")[offset:]
        ld.ld_pack_planes(sim.ctx, z0, count, buf)
        idx = [(z0 + k) % nz for k in range(count)]
        got = buf.view(38, count, ny, nx)
        # distributions() decodes: compare through a second lattice that unpacks the planes into other contents
        other = ld.LdSim(nx, ny, nz, precision=precision)
        other.set_distributions(g, f)
        before = torch.cat(other.distributions())
        ld.ld_unpack_planes(other.ctx, z0, count, got)
        after = torch.cat(other.distributions())
        assert torch.equal(after[:, idx], state[:, idx])
        rest = [z for z in range(nz) if z not in idx]
        assert torch.equal(after[:, rest], before[:, rest])


def test_planes_in_a_graph():
    """Both copies under stream capture, on a stream of their own; a replay copies the state of its time."""
    nx, ny, nz = 9, 5, 8
    sim = ld.LdSim(nx, ny, nz, precision="fp32")
    stream = torch.cuda.Stream()
    ld.ld_set_stream(sim.ctx, stream.cuda_stream)
    f, g = torch.rand((2, 19, nz, ny, nx), dtype=torch.float64, device="cuda")
    buf = torch.empty((38, 2, ny, nx), dtype=torch.float32, device="cuda")
    stream.wait_stream(torch.cuda.current_stream())
    sim.set_distributions(f, g)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ld.ld_pack_planes(sim.ctx, 1, 2, buf)
        ld.ld_unpack_planes(sim.ctx, 5, 2, buf)
    with torch.cuda.stream(stream):
        sim.set_distributions(g, f)
        graph.replay()
        after = torch.cat(sim.distributions())
    stream.synchronize()
    want = torch.cat((g, f)).float().double()
    want[:, 5:7] = want[:, 1:3]
    assert torch.equal(after, want)

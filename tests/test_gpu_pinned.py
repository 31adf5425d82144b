"""3D retrieval and refinement into pinned host memory, written in place or decoded
on the device and copied: boxes around the sizes where that changes (2, 4 and 8
MiB), rows of whole 16-byte words and others, buffers at any alignment of their
type; and under stream capture."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MIB = 1 << 20


def _field(shape, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(51)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nx", [64, 65, 66])
def test_pinned_boxes_of_every_route(dtype, nx):
    import paper_2308_11759_gb300 as P

    width = torch.finfo(dtype).bits // 8
    nz = 9 * MIB // (64 * 64 * width) + 1
    x = _field((nz, 64, nx), dtype)
    st = P.compress(x, [0.25, 2.0 ** -6, 2.0 ** -10])
    for size in (2, 4, 8):
        most = -(-size * MIB // (64 * nx * width))  # planes of `size` MiB, rounded up
        for z in (most - 1, most):
            box = ([1, 0, 0], [1 + z, 64, nx])
            want = [st.retrieve(k=k, box=box) for k in (1, 3)]
            for off in (0, 1):
                host = torch.full((z * 64 * nx + 2,), 7, dtype=dtype).pin_memory()
                out = host[off:off + z * 64 * nx].view(z, 64, nx)
                st.retrieve(k=1, box=box, out=out)
                torch.cuda.synchronize()
                assert torch.equal(out, want[0].cpu())
                st.refine(1, 3, out, box=box)
                torch.cuda.synchronize()
                assert torch.equal(out, want[1].cpu())
                assert (host[:off] == 7).all() and (host[off + z * 64 * nx:] == 7).all()


def test_pinned_result_under_capture():
    import paper_2308_11759_gb300 as P

    x = _field((70, 81, 83), torch.float64)
    st = P.compress(x, [0.25, 2.0 ** -6])
    want = st.retrieve(k=2).cpu()
    out = torch.zeros(x.shape, dtype=torch.float64).pin_memory()
    st.retrieve(k=2, out=out)
    torch.cuda.synchronize()
    out.zero_()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        st.retrieve(k=2, out=out, stream=stream)
    assert not out.any()
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    assert np.array_equal(out.numpy(), want.numpy())

"""jdft_subspace of FP64 blocks uses nothing that two calls could share: calls of one basis on two streams, and calls
under stream capture, give what one call by itself gives."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _basis():
    from paper_1708_03621_gb300 import jdft
    return jdft, jdft.Basis(np.eye(3) * 10.0, (48, 48, 48), 20.0, [(0.1, 0.2, 0.3)])


def _block(nb, npw, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn((nb, npw, 2), generator=g, dtype=torch.float64, device="cuda"))


def test_two_streams():
    jdft, b = _basis()
    sizes = (128, 96)
    blocks = [_block(nb, b.npw(0), nb) for nb in sizes]
    refs = []
    for C in blocks:
        M = torch.empty((len(C), len(C)), dtype=torch.complex128, device="cuda")
        jdft.jdft_subspace(b, 0, C, None, None, M)
        torch.cuda.synchronize()
        refs.append(M)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [[torch.zeros_like(r) for _ in range(20)] for r in refs]
    torch.cuda.synchronize()
    for i in range(20):
        for C, st, out in zip(blocks, streams, outs):
            jdft.jdft_subspace(b, 0, C, None, None, out[i], stream=st)
    torch.cuda.synchronize()
    jdft.jdft_device_status()
    for out, ref in zip(outs, refs):
        assert all(torch.equal(o, ref) for o in out)


@pytest.mark.parametrize("warm", [False, True])
def test_capture(warm):
    """The first FP64 call of a basis may be one under capture; the bound is that of the FP64 products' sums, npw units
    of 2^-53 of the rows' norms (which differ by a few per cent)."""
    jdft, b = _basis()
    nb, npw = 96, b.npw(0)
    C = _block(nb, npw, 3)
    M = torch.zeros((nb, nb), dtype=torch.complex128, device="cuda")
    if warm:
        jdft.jdft_subspace(b, 0, C, None, None, M)
        M.zero_()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        jdft.jdft_subspace(b, 0, C, None, None, M)
    ref = 1000.0 * (C.conj() @ C.T)
    for seed in (3, 4):
        C.copy_(_block(nb, npw, seed))
        ref = 1000.0 * (C.conj() @ C.T)
        graph.replay()
        torch.cuda.synchronize()
        assert float((M - ref).abs().max() / ref.abs().max()) <= npw * 2.0 ** -53

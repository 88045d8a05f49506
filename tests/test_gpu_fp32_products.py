"""FP32 products on the CUDA cores (gemm.cu) at the edges of their tiles, against FP64.

Bounds (derived before the first run), relative to the sums of absolute products, in units of 2^-24.  conj(A) B: a split of
K holds at most 144 values here, two products each in one FP32 chain: 300.  The projector term has that, the rounding of
D P^dag C, and a chain of two products per projector (at most 66): 300 + 1 + 140 < 512, and one rounding of H C itself.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _setup(nb):
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * 10.0, (48, 48, 48), 20.0, [(0.1, 0.2, 0.3)])
    rng = np.random.default_rng(nb)
    C = (rng.standard_normal((nb, b.npw(0))) + 1j * rng.standard_normal((nb, b.npw(0)))).astype(np.complex64)
    return jdft, b, rng, C


@pytest.mark.parametrize("nb", [1, 31, 33, 65, 155, 161])
def test_subspace_entries(nb):
    jdft, b, rng, C = _setup(nb)
    H = (rng.standard_normal(C.shape) + 1j * rng.standard_normal(C.shape)).astype(np.complex64)
    out = torch.empty((2, nb, nb), dtype=torch.complex128, device="cuda")
    jdft.jdft_subspace(b, 0, torch.tensor(C, device="cuda"), torch.tensor(H, device="cuda"), out[0], out[1], prec="fp32")
    c, h = C.astype(np.complex128), H.astype(np.complex128)
    for got, x, s in ((out[0].cpu().numpy(), h, 1.0), (out[1].cpu().numpy(), c, 1000.0)):
        assert np.all(np.abs(got - s * (c.conj() @ x.T)) <= 300 * U * s * (np.abs(c) @ np.abs(x).T))


@pytest.mark.parametrize("nb, nproj", [(15, 33), (40, 7), (289, 33), (300, 17)])
def test_projector_term(nb, nproj):
    jdft, b, rng, C = _setup(nb)
    npw = C.shape[1]
    P = (rng.standard_normal((nproj, npw)) + 1j * rng.standard_normal((nproj, npw))).astype(np.complex64)
    P = P.astype(np.complex128)
    dd = rng.uniform(-1, 1, nproj)
    jdft.jdft_set_potential(b, torch.zeros(48 ** 3, dtype=torch.float64, device="cuda"))
    Cd = torch.tensor(C, device="cuda")
    H0, HC = torch.empty_like(Cd), torch.empty_like(Cd)
    jdft.jdft_apply_H(b, 0, Cd, H0, prec="fp32")
    jdft.jdft_set_projectors(b, 0, torch.tensor(P, device="cuda"), torch.tensor(np.diag(dd), device="cuda"))
    jdft.jdft_apply_H(b, 0, Cd, HC, prec="fp32")
    c = C.astype(np.complex128)
    ref = H0.cpu().numpy().astype(np.complex128) + ((P.conj() @ c.T) * dd[:, None]).T @ P
    scale = ((np.abs(P) @ np.abs(c).T) * np.abs(dd)[:, None]).T @ np.abs(P)
    assert np.all(np.abs(HC.cpu().numpy() - ref) <= 512 * U * scale + U * np.abs(ref) * 2)

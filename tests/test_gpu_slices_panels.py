"""Sliced FP64 products larger than their scratch budget: panels of the summed index and of both outputs' sides."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches(jdft, call):
    jdft.jdft_profile_enable(True)
    jdft.jdft_profile_read()
    call()
    torch.cuda.synchronize()
    names = jdft.jdft_profile_read()
    jdft.jdft_profile_enable(False)
    return names


def _block(nb, npw, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn((nb, npw, 2), generator=g, dtype=torch.float64, device="cuda"))


def test_panels_of_the_summed_index():
    """C^dag H C of 200 bands and 62 759 plane waves: two operands' slices exceed the budget, so two panels are summed.
    Against torch's FP64 product, both within npw units of 2^-53 of the rows' norms in the worst case and some sqrt(npw)
    in earnest: 1e-14 of the largest entry (62 759 x 2^-53 is 7e-12)."""
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * 20.0, (128, 128, 128), 30.0, [(0.1, 0.2, 0.3)])
    nb = 200
    C = _block(nb, b.npw(0), 3)
    H = _block(nb, b.npw(0), 4) + C
    out = torch.empty((nb, nb), dtype=torch.complex128, device="cuda")
    names = _launches(jdft, lambda: jdft.jdft_subspace(b, 0, C, H, out, None))
    assert names["sl_mma"][0] == 2 and "zgemm_cn" not in names
    ref = C.conj() @ H.T
    assert float((out - ref).abs().max() / ref.abs().max()) < 1e-14


def test_scratch_stays_within_its_bound():
    """Subspace matrices of 4096 bands, and H C of 4096 bands with 4096 projectors, on 4 259 plane waves: the device
    holds at most 1 GiB of scratch for either call (and an outgrown block, for the second product of H C), and beside
    it what the calls need otherwise (below 1 GiB of basis workspace for H C).  Sampled entries against torch's FP64 products, in units of the sums' worst case."""
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * 10.0, (48, 48, 48), 20.0, [(0.1, 0.2, 0.3)])
    n, npw, u = 4096, b.npw(0), 2.0 ** -53
    jdft.jdft_set_potential(b, torch.zeros(48 ** 3, dtype=torch.float64, device="cuda"))
    C, P = _block(n, npw, 5), _block(n, npw, 6)
    D = torch.diag(torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda"))
    H0, HC = torch.empty_like(C), torch.empty_like(C)
    out = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    jdft.jdft_apply_H(b, 0, C[:64], H0[:64])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    names = _launches(jdft, lambda: jdft.jdft_subspace(b, 0, C, P, out, None))
    assert "zgemm_cn" not in names
    assert free - torch.cuda.mem_get_info()[0] <= (1 << 30) + (32 << 20)
    ref = C[:64].conj() @ P.T
    assert float((out[:64] - ref).abs().max()) <= npw * u * float(C.abs().max() * P.abs().max()) * 4
    jdft.jdft_set_projectors(b, 0, None, None)
    jdft.jdft_apply_H(b, 0, C, H0)
    jdft.jdft_set_projectors(b, 0, P, D)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    names = _launches(jdft, lambda: jdft.jdft_apply_H(b, 0, C, HC))
    assert "zgemm_nn" not in names and "zgemm_cn" not in names
    assert free - torch.cuda.mem_get_info()[0] <= 3 << 30
    PC = D.diagonal()[:, None] * (P.conj() @ C[-64:].T)
    ref = H0[-64:] + (P.T @ PC).T
    scale = float((P.abs().max() * PC.abs().max()) * n)
    assert float((HC[-64:] - ref).abs().max()) <= 64 * u * scale

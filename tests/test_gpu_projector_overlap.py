"""P^dag C on the CUDA cores beside the FFT chain, P (D P^dag C) on the CUDA cores or from slices, against long double.

Bound (derived before the first run), relative to the products of absolute values: a projection adds at most 32 fused
products in a lane, four warps' sums and one sum per block of K (at most 152 blocks, of 28 for one tile), the second product
at most 2 x 36 of them in sequence and one addition: below 256 units of 2^-53.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("nb, nproj, sliced", [(1, 1, 0), (13, 32, 0), (17, 36, 0), (61, 32, 1), (64, 32, 1)])
def test_projections_beside_the_chain(nb, nproj, sliced):
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * 10.0, (48, 48, 48), 20.0, [(0.1, 0.2, 0.3)])
    npw = b.npw(0)
    rng = np.random.default_rng(nb)
    P = rng.standard_normal((nproj, npw)) + 1j * rng.standard_normal((nproj, npw))
    C = rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))
    dd = rng.uniform(-1, 1, nproj)
    jdft.jdft_set_potential(b, torch.zeros(48 ** 3, dtype=torch.float64, device="cuda"))
    Cd = torch.tensor(C, device="cuda")
    H0, HC = torch.empty_like(Cd), torch.empty_like(Cd)
    jdft.jdft_apply_H(b, 0, Cd, H0)
    jdft.jdft_set_projectors(b, 0, torch.tensor(P, device="cuda"), torch.tensor(np.diag(dd), device="cuda"))
    jdft.jdft_profile_enable(True)
    jdft.jdft_profile_read()
    jdft.jdft_apply_H(b, 0, Cd, HC)
    torch.cuda.synchronize()
    names = jdft.jdft_profile_read()
    jdft.jdft_profile_enable(False)
    assert names["zgemm_cn"][0] == 1 and ("sl_mma" in names) == bool(sliced) and ("zgemm_nn" in names) == (not sliced)
    ld = np.clongdouble
    PC = (P.conj().astype(ld) @ C.T.astype(ld)) * dd[:, None]
    cols = [0, 1, npw // 2, npw - 1]
    ref = H0.cpu().numpy().astype(ld)[:, cols] + (P.T.astype(ld)[cols] @ PC).T
    scale = (np.abs(P.T[cols]) @ (np.abs(P) @ np.abs(C).T * np.abs(dd)[:, None])).T
    assert np.all(np.abs(HC.cpu().numpy()[:, cols] - ref) <= 256 * U * scale + 3 * U * np.abs(ref))

"""FP64 products from 7-bit slices on the tensor cores (tc_slices.cuh) against extended precision.

Bound for an entry sum_k conj(a_k) b_k (derived before the first run): what the slices drop is below 2^-60 of the two
rows' largest components per real product, so K 2^-58 max|a| max|b| over the two products of a component with room for
their sum; the integer sum is rounded once, scaled and added once: 3 units of 2^-53 of the entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _basis(L=10.0, S=48, ecut=20.0):
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * L, (S, S, S), ecut, [(0.1, 0.2, 0.3)])
    return jdft, b, b.npw(0)


def _block(rng, nb, npw, ld, spread=3.0):
    C = np.zeros((nb, ld), dtype=np.complex128)
    C[:, :npw] = rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))
    C[:, :npw] *= 10.0 ** rng.uniform(-spread, 0, (nb, npw))
    C[:, npw:] = np.nan  # never read
    return C


def _subspace(jdft, b, C, H):
    nb = C.shape[0]
    Cd, Hd = torch.tensor(C, device="cuda"), torch.tensor(H, device="cuda")
    out = torch.empty((2, nb, nb), dtype=torch.complex128, device="cuda")
    jdft.jdft_profile_enable(True)
    jdft.jdft_profile_read()
    jdft.jdft_subspace(b, 0, Cd, Hd, out[0], out[1])
    torch.cuda.synchronize()
    names = jdft.jdft_profile_read()
    jdft.jdft_profile_enable(False)
    jdft.jdft_device_status()
    return out[0].cpu().numpy(), out[1].cpu().numpy(), names


@pytest.mark.parametrize("nb, pad", [(48, 0), (64, 1), (65, 0), (96, 5), (128, 0), (130, 3)])
def test_subspace_entries(nb, pad):
    jdft, b, npw = _basis()
    rng = np.random.default_rng(nb)
    C, H = _block(rng, nb, npw, npw + pad), _block(rng, nb, npw, npw + pad)
    chc, coc, names = _subspace(jdft, b, C, H)
    assert "sl_mma" in names and "zgemm_cn" not in names
    om = 1000.0
    ld = np.clongdouble
    c, h = C[:, :npw].astype(ld), H[:, :npw].astype(ld)
    ma = np.maximum(np.abs(C[:, :npw].real), np.abs(C[:, :npw].imag)).max(1)
    mh = np.maximum(np.abs(H[:, :npw].real), np.abs(H[:, :npw].imag)).max(1)
    for m in (0, 1, nb // 2, nb - 1):
        for got, other, mo, s in ((chc, h, mh, 1.0), (coc, c, ma, om)):
            ref = s * (c[m].conj()[None, :] * other).sum(1)
            tol = 3 * U * np.abs(ref) + s * npw * 2.0 ** -58 * ma[m] * mo
            for part in ("real", "imag"):
                e = np.abs(getattr(got[m], part) - getattr(ref, part))
                assert np.all(e <= tol), (m, float((e / tol).max()))


def test_largest_digit_sums_are_exact():
    """Rows of one value whose digits are almost all -64: sums of 2^23 and more in tensor memory."""
    jdft, b, npw = _basis()
    x = -(32 * 2 ** 56 + sum(64 * 2 ** (7 * j) for j in range(2, 8)))
    nb = 64
    C = np.full((nb, npw), complex(float(x), float(x)))
    chc, coc, names = _subspace(jdft, b, C, C)
    assert "sl_mma" in names
    exact = 2 * npw * x * x
    assert np.all(np.abs(chc.real / float(exact) - 1.0) <= 2 * U)
    assert np.all(chc.imag == 0.0)


def test_scales_and_non_finite_rows():
    jdft, b, npw = _basis()
    rng = np.random.default_rng(5)
    nb = 64
    C, H = _block(rng, nb, npw, npw), _block(rng, nb, npw, npw)
    ref = _subspace(jdft, b, C, H)[0]
    D = C.copy()
    D[3] = np.ldexp(C[3].real, -1010) + 1j * np.ldexp(C[3].imag, -1010)  # many of its values denormal
    D[7] = np.ldexp(C[7].real, 700) + 1j * np.ldexp(C[7].imag, 700)
    D[9] = 0.0
    D[11, 17] = np.nan
    D[12, 5] = np.inf
    got = _subspace(jdft, b, D, H)[0]
    same = [i for i in range(nb) if i not in (3, 7, 9, 11, 12)]
    assert np.array_equal(got[same], ref[same])
    assert np.array_equal(got[7], np.ldexp(ref[7].real, 700) + 1j * np.ldexp(ref[7].imag, 700))
    assert np.all(got[9] == 0.0) and np.isnan(got[11]).all() and np.isnan(got[12]).all()
    # denormal values keep 2^-1074: relative to the row's largest, 2^-1010 and up, 2^-64 each
    scale = np.abs(C[3]).max() * np.abs(H).max(1) * npw
    assert np.all(np.abs(np.ldexp(got[3].real, 1010) - ref[3].real) <= 2.0 ** -50 * scale)


@pytest.mark.parametrize("nb, natoms", [(40, 10), (65, 33), (24, 64)])
def test_projector_products(nb, natoms):
    """P D P^dag C alone (V = 0), out of both products, against long double."""
    jdft, b, npw = _basis()
    rng = np.random.default_rng(nb)
    nproj = 4 * natoms
    P, C = _block(rng, nproj, npw, npw, 1.0), _block(rng, nb, npw, npw, 1.0)
    dd = rng.uniform(-1, 1, nproj)
    jdft.jdft_set_potential(b, torch.zeros(48 ** 3, dtype=torch.float64, device="cuda"))
    Cd = torch.tensor(C, device="cuda")
    jdft.jdft_set_projectors(b, 0, None, None)
    H0 = torch.empty_like(Cd)
    jdft.jdft_apply_H(b, 0, Cd, H0)
    jdft.jdft_set_projectors(b, 0, torch.tensor(P, device="cuda"), torch.tensor(np.diag(dd), device="cuda"))
    HC = torch.empty_like(Cd)
    jdft.jdft_profile_enable(True)
    jdft.jdft_profile_read()
    jdft.jdft_apply_H(b, 0, Cd, HC)
    torch.cuda.synchronize()
    names = jdft.jdft_profile_read()
    jdft.jdft_profile_enable(False)
    assert names["sl_mma"][0] == 2
    ld = np.clongdouble
    PC = (P.conj().astype(ld) @ C.T.astype(ld)) * dd[:, None]
    cols = [0, 1, npw // 2, npw - 1]
    ref = H0.cpu().numpy().astype(ld)[:, cols] + (P.T.astype(ld)[cols] @ PC).T
    got = HC.cpu().numpy()[:, cols]
    # the projections carry a few units each, and the second product's bound comes on top of the sums' rounding
    scale = (np.abs(P.T[cols]) @ (np.abs(P) @ np.abs(C).T * np.abs(dd)[:, None])).T
    assert np.all(np.abs(got - ref) <= 8 * U * scale + 3 * U * np.abs(ref))


def test_panels_of_a_large_product_match():
    """A block whose slices exceed the scratch budget runs in panels; sampled entries against FP64 sums."""
    jdft, b, npw = _basis(20.0, 128, 30.0)
    rng = np.random.default_rng(1)
    nb = 200
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    C = torch.randn((nb, npw, 2), generator=g, dtype=torch.float64, device="cuda")
    C = torch.view_as_complex(C)
    out = torch.empty((nb, nb), dtype=torch.complex128, device="cuda")
    jdft.jdft_subspace(b, 0, C, None, None, out)
    ref = 8000.0 * (C.conj() @ C.T)
    torch.cuda.synchronize()
    assert float((out - ref).abs().max() / ref.abs().max()) < 1e-14
    D = C.clone()
    jdft.jdft_orthonormalize(b, 0, D)
    eye = 8000.0 * (D.conj() @ D.T)
    assert float((eye - torch.eye(nb, device="cuda")).abs().max()) < 1e-12
    del rng

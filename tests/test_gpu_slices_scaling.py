"""Sliced FP64 products (tc_slices.cuh) of badly scaled operands: bands or projectors whose norms differ by many
orders of magnitude, and coefficients and H C that grow and decay oppositely over the plane waves.

What the products replace rounds every term to 2^-53 of itself, so no scaling of the summed index shows in it.
Bounds are derived before the first run, in each test's docstring; references are long double.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
LD = np.clongdouble


def _basis(L=10.0, S=48, ecut=20.0):
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * L, (S, S, S), ecut, [(0.1, 0.2, 0.3)])
    return jdft, b, b.npw(0)


def _normal(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _profiled(jdft, call):
    jdft.jdft_profile_enable(True)
    jdft.jdft_profile_read()
    call()
    torch.cuda.synchronize()
    names = jdft.jdft_profile_read()
    jdft.jdft_profile_enable(False)
    return names


def _power(rng, spread, n):
    """n powers of two spread over 10^-spread .. 1, both ends taken, in random order."""
    e = -np.round(np.linspace(0.0, spread * np.log2(10.0), n)).astype(int)
    return np.ldexp(1.0, rng.permutation(e))


@pytest.mark.parametrize("nb", [64, 96])
@pytest.mark.parametrize("spread", [0, 6, 12, 20, 100])
def test_orthonormalize_bands_of_different_norms(nb, spread):
    """C L^-dag is invariant under a scaling of the bands.  The normalised bands' overlap has condition below 2
    (random vectors, nb << npw); overlap, factor, inverse and product err by at most about nb units of 2^-53 each:
    16 nb U with that condition and room for two."""
    jdft, b, npw = _basis()
    rng = np.random.default_rng(nb + spread)
    C = _normal(rng, nb, npw) * _power(rng, spread, nb)[:, None]
    Cd = torch.tensor(C, device="cuda")
    names = _profiled(jdft, lambda: jdft.jdft_orthonormalize(b, 0, Cd))
    assert names["sl_mma"][0] == 2
    D = Cd.cpu().numpy().astype(LD)
    eye = 1000.0 * (D.conj() @ D.T)
    assert np.abs(eye - np.eye(nb)).max() <= 16 * nb * U


@pytest.mark.parametrize("spread", [0, 6, 20])
def test_projectors_of_different_norms(spread):
    """P D P^dag C with P_i scaled by s_i and D_i by s_i^-2: the same operator.  Entries against the sum of absolute
    values of the terms, 8 units of 2^-53 of it (a few for the projections, one for the second product's rounding)
    and 3 of the entry."""
    jdft, b, npw = _basis()
    rng = np.random.default_rng(17 + spread)
    nb, nproj = 40, 132
    P, C = _normal(rng, nproj, npw), _normal(rng, nb, npw)
    s = _power(rng, spread, nproj)
    P *= s[:, None]
    dd = rng.uniform(-1, 1, nproj) / s ** 2
    jdft.jdft_set_potential(b, torch.zeros(48 ** 3, dtype=torch.float64, device="cuda"))
    jdft.jdft_set_projectors(b, 0, None, None)
    Cd = torch.tensor(C, device="cuda")
    H0, HC = torch.empty_like(Cd), torch.empty_like(Cd)
    jdft.jdft_apply_H(b, 0, Cd, H0)
    jdft.jdft_set_projectors(b, 0, torch.tensor(P, device="cuda"), torch.tensor(np.diag(dd), device="cuda"))
    names = _profiled(jdft, lambda: jdft.jdft_apply_H(b, 0, Cd, HC))
    assert names["sl_mma"][0] == 2
    cols = [0, 1, npw // 2, npw - 1]
    PC = (P.conj().astype(LD) @ C.T.astype(LD)) * dd[:, None]
    ref = H0.cpu().numpy().astype(LD)[:, cols] + (P.T.astype(LD)[cols] @ PC).T
    got = HC.cpu().numpy()[:, cols]
    scale = (np.abs(P.T[cols]) @ (np.abs(P) @ np.abs(C).T * np.abs(dd)[:, None])).T
    assert np.all(np.abs(got - ref) <= 8 * U * scale + 3 * U * np.abs(ref))


@pytest.mark.parametrize("nb, spread, norms", [(64, 0, 0), (64, 6, 0), (96, 10, 0), (64, 10, 8), (96, 40, 20)])
def test_subspace_of_oppositely_graded_blocks(nb, spread, norms):
    """C^dag H C where C falls by 10^spread over the plane waves (in random order) and H C rises by as much, bands of
    different norms among them: every term is of one size, far below the product of the rows' maxima.  With r the rows'
    largest components and a_k, b_k the columns' largest relative to them, the scaled rows stay below 2 sqrt(a_k b_k)
    r each (halves and exponents rounded down), and each real product loses 2^-58 of their maxima to the cut and 2^-56
    in the digit pairs left out: npw 2^-53 max(a_k b_k) r r' for a component's two, of either sign.  Half of that is
    asked for, and the entry is rounded three times."""
    jdft, b, npw = _basis()
    rng = np.random.default_rng(nb + spread + norms)
    x = _power(rng, spread, npw)[None, :]
    s = _power(rng, norms, nb)[:, None]
    C, H = _normal(rng, nb, npw) * x * s, _normal(rng, nb, npw) / x / s
    out = torch.empty((nb, nb), dtype=torch.complex128, device="cuda")
    Cd, Hd = torch.tensor(C, device="cuda"), torch.tensor(H, device="cuda")
    names = _profiled(jdft, lambda: jdft.jdft_subspace(b, 0, Cd, Hd, out, None))
    assert names["sl_mma"][0] == 1
    got = out.cpu().numpy()
    ref = C.conj().astype(LD) @ H.astype(LD).T
    big = [np.maximum(np.abs(z.real), np.abs(z.imag)) for z in (C, H)]
    r = [z.max(1) for z in big]
    a, bk = ((z / q[:, None]).max(0) for z, q in zip(big, r))
    tol = npw * 2.0 ** -54 * (a * bk).max() * r[0][:, None] * r[1][None, :]
    assert np.all(np.abs(got.real - ref.real) <= tol + 3 * U * np.abs(ref))
    assert np.all(np.abs(got.imag - ref.imag) <= tol + 3 * U * np.abs(ref))


def test_rotation_keeps_a_non_finite_coefficient_to_its_plane_wave():
    """With the overlap given, a NaN or infinity among the coefficients of one plane wave reaches that plane wave's
    outputs only; the others are the same bits."""
    jdft, b, npw = _basis()
    rng = np.random.default_rng(5)
    nb = 64
    C = _normal(rng, nb, npw) * _power(rng, 12, nb)[:, None]
    C[:, 100] *= 1e-3  # not the largest of any band
    Ov = torch.tensor(1000.0 * (C.conj() @ C.T), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs = []
    for bad in (None, np.nan, np.inf):
        D = C.copy()
        if bad is not None:
            D[3, 100] = bad
        Dd = torch.tensor(D, device="cuda")
        names = _profiled(jdft, lambda: jdft.jdft_orthonormalize_async(b, 0, Dd, status, U=Ov))
        assert names["sl_mma"][0] == 1
        outs.append(Dd.cpu().numpy())
    rest = [k for k in range(npw) if k != 100]
    for o in outs[1:]:
        assert np.array_equal(o[:, rest], outs[0][:, rest])
        assert not np.isfinite(o[:, 100]).any()

"""The fixed-point line transforms behind FP64 blocks (fft_fix.cuh) against extended precision.

H C without projectors (I, multiply by V, J and the kinetic term) on boxes of every compiled line length, against the
same chain in numpy's long double.  The tolerance is 8 units of 2^-53 of the result's norm: six line passes, each
rounded to FP64 on the way out (0.6 units) with at most half a unit from the fixed-point roundings, and the products
with V and the kinetic energy (one unit each), added in quadrature, with a factor of two to spare.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 8 * 2.0 ** -53

# box, cell edges: the sphere at E_cut fits the box
SHAPES = [
    ((12, 12, 12), (6.0, 6.0, 6.0), 4.0),
    ((16, 12, 16), (7.0, 5.0, 7.0), 5.0),
    ((40, 40, 40), (9.0, 9.0, 9.0), 14.0),
    ((48, 48, 48), (10.0, 10.0, 10.0), 20.0),
    ((64, 64, 64), (15.0, 15.0, 15.0), 20.0),
    ((80, 80, 80), (18.0, 18.0, 18.0), 20.0),
    ((128, 128, 40), (20.0, 20.0, 6.0), 30.0),
    ((256, 128, 12), (40.0, 20.0, 1.6), 30.0),
    ((12, 12, 256), (1.6, 1.6, 40.0), 30.0),
]


def _system(shape, nb=2, seed=3):
    from paper_1708_03621_gb300 import jdft
    S, L, ecut = shape
    b = jdft.Basis(np.diag(L), S, ecut, [(0.1, 0.2, 0.3)])
    g = b.gvectors(0).astype(np.int64)
    rng = np.random.default_rng(seed)
    q = (g + np.array([0.1, 0.2, 0.3])) * (2 * np.pi / np.array(L))
    C = (rng.standard_normal((nb, len(g))) + 1j * rng.standard_normal((nb, len(g)))) / (1 + (q * q).sum(1))
    V = -3.0 * rng.random(S) + 0.5
    jdft.jdft_set_potential(b, torch.tensor(V.reshape(-1), device="cuda"))
    return jdft, b, g, q, C, V


def _apply(jdft, b, C):
    Cd = torch.tensor(C, device="cuda")
    HC = torch.empty_like(Cd)
    jdft.jdft_apply_H(b, 0, Cd, HC)
    torch.cuda.synchronize()
    return HC.cpu().numpy()


def _reference(S, L, g, q, C, V):
    import scipy.fft
    ld = np.clongdouble
    slot = ((g[:, 0] % S[0]) * S[1] + g[:, 1] % S[1]) * S[2] + g[:, 2] % S[2]
    box = np.zeros((len(C), int(np.prod(S))), dtype=ld)
    box[:, slot] = C
    psi = scipy.fft.ifftn(box.reshape((-1,) + S), axes=(1, 2, 3), norm="forward")
    assert psi.dtype == ld
    back = scipy.fft.fftn(psi * V.astype(np.longdouble), axes=(1, 2, 3), norm="forward").reshape(len(C), -1)[:, slot]
    # k+G from the library's B = 2 pi R^-T in FP64, as the kinetic table is FP64
    T = (0.5 * (q * q).sum(1)).astype(np.longdouble)
    return np.longdouble(np.prod(L)) * (T * C.astype(ld) + back)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s[0])))
def test_error_against_extended_precision(shape):
    jdft, b, g, q, C, V = _system(shape)
    # a band whose values span forty orders of magnitude, and one with a single plane wave
    C = np.concatenate([C, C[:1] * 10.0 ** np.linspace(0, -40, C.shape[1]), np.zeros_like(C[:1])])
    C[3, len(g) // 3] = 0.3 - 1.7j
    ref = _reference(shape[0], shape[1], g, q, C, V)
    got = _apply(jdft, b, C)
    err = np.sqrt((np.abs(got - ref) ** 2).sum(1) / (np.abs(ref) ** 2).sum(1)).astype(float)
    assert np.all(err < TOL), err / 2.0 ** -53


@pytest.mark.parametrize("shape", [SHAPES[1], SHAPES[3], SHAPES[6]], ids=lambda s: "x".join(map(str, s[0])))
def test_power_of_two_scales_and_non_finite_bands(shape):
    jdft, b, g, q, C, V = _system(shape)
    ref = _apply(jdft, b, C)
    for p in (-600, 500):
        assert np.array_equal(_apply(jdft, b, np.ldexp(C.real, p) + 1j * np.ldexp(C.imag, p)),
                              np.ldexp(ref.real, p) + 1j * np.ldexp(ref.imag, p))
    # values near the bottom of the range, where the lines are scaled up first
    tiny = _apply(jdft, b, np.ldexp(C.real, -980) + 1j * np.ldexp(C.imag, -980))
    back = np.ldexp(tiny.real, 980) + 1j * np.ldexp(tiny.imag, 980)
    assert np.linalg.norm(back - ref) < 2.0 ** -40 * np.linalg.norm(ref)
    assert np.array_equal(_apply(jdft, b, 0 * C), 0 * C)
    for bad in (np.nan, np.inf):
        D = C.copy()
        D[0, 5] = bad
        got = _apply(jdft, b, D)
        assert np.isnan(got[0]).all() and np.array_equal(got[1], ref[1])

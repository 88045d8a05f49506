"""Register-FFT field transforms (field_fast.cuh) on every compiled length, in skewed cells, and the point-wise LDA,
against the same formulas in numpy's long double (the oracle's FP64 transforms are themselves 100 units off where the
mean density dominates).

Tolerances (relative to the result's norm): a transform pass carries about one unit u = 2^-53 (rounding on the way out and
the fixed-point roundings); 32 u for chains of three to six passes and 64 u where the G = 0 term that is dropped dominates
the input.  LDA: 16 u of the value for some thirty FP64 operations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53
LD = np.longdouble
SKEW = np.array([[7.0, 1.1, -0.6], [0.4, 6.2, 0.9], [0.0, -0.7, 8.1]])
BOXES = [(12, 16, 40), (40, 12, 16), (16, 48, 12), (48, 40, 64), (64, 12, 80), (80, 64, 12), (12, 128, 16), (16, 12, 256),
         (256, 16, 12), (128, 12, 48)]
# the other lengths, each on every axis
_REST = [24, 25, 27, 30, 32, 36, 45, 50, 54, 60, 72, 75, 81, 90, 96, 100, 108, 120, 125]
RAGGED = [(_REST[i], _REST[(i + 7) % 19], _REST[(i + 13) % 19]) for i in range(19)]


def _basis(S):
    from paper_1708_03621_gb300 import jdft
    return jdft, jdft.Basis(SKEW, S, 0.2, [(0.0, 0.0, 0.0)])


def _G(S):
    """Cartesian G of every slot (folded frequencies), long double."""
    ax = [np.fft.fftfreq(s, 1 / s).round() for s in S]
    g = np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3).astype(LD)
    return g @ (2 * np.pi * np.linalg.inv(SKEW).T).T.astype(LD)


def _I(S, X):
    import scipy.fft
    return scipy.fft.ifftn(np.asarray(X).astype(np.clongdouble).reshape(S), norm="forward").reshape(-1)


def _J(S, x):
    import scipy.fft
    return scipy.fft.fftn(np.asarray(x).astype(np.clongdouble).reshape(S), norm="forward").reshape(-1)


def _coulomb(S):
    G2 = (_G(S) ** 2).sum(1)
    return np.where(G2 > 0, LD("12.566370614359172953850573533118") / np.where(G2 > 0, G2, 1), 0)


def _hessian(S, eps, x):
    G = _G(S)
    out = sum(1j * G[:, d] * _J(S, eps * _I(S, 1j * G[:, d] * x)) for d in range(3))
    return -out / LD("12.566370614359172953850573533118")


def _lda(n):
    """(e_xc, v_xc) in long double."""
    x = np.asarray(n).astype(LD)
    e, v = np.zeros_like(x), np.zeros_like(x)
    pos = x > 0
    c = x[pos] ** (LD(1) / 3)
    pi = LD("3.14159265358979323846264338327950288")
    ex = -LD(3) / 4 * (3 / pi) ** (LD(1) / 3) * c
    rs = (3 / (4 * pi)) ** (LD(1) / 3) / c
    g, b1, b2, A, B, C, D = (LD(s) for s in ("-0.1423", "1.0529", "0.3334", "0.0311", "-0.048", "0.0020", "-0.0116"))
    sq, lr = np.sqrt(rs), np.log(rs)
    den = 1 + b1 * sq + b2 * rs
    hi = rs >= 1
    ec = np.where(hi, g / den, A * lr + B + C * rs * lr + D * rs)
    rd = np.where(hi, -g * (b1 * sq / 2 + b2 * rs) / den ** 2, A + rs * (C * (lr + 1) + D))
    e[pos], v[pos] = ex + ec, 4 * ex / 3 + ec - rd / 3
    return e, v


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("S", BOXES, ids=lambda s: "x".join(map(str, s)))
def test_transforms_and_hartree(S):
    jdft, b = _basis(S)
    N = int(np.prod(S))
    rng = np.random.default_rng(N)
    x = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    xd = torch.tensor(x, device="cuda")
    out = torch.empty_like(xd)
    jdft.jdft_field_I(b, xd, out)
    assert _rel(out.cpu().numpy(), _I(S, x)) < 32 * U64
    jdft.jdft_field_J(b, xd, xd)  # in place
    assert _rel(xd.cpu().numpy(), _J(S, x)) < 32 * U64
    # a density with weight on the Nyquist planes, where the two mirror slots differ in a skewed cell
    n = 0.05 * rng.random(N) + 1e-3
    vion = rng.standard_normal(N)
    K, nt, om = _coulomb(S), _J(S, n), LD(np.linalg.det(SKEW))
    vh = _I(S, K * nt).real
    eh = float(om / 2 * (K * np.abs(nt) ** 2).sum())
    exc_n, vxc = _lda(n)
    exc, vks = float(om / N * (n * exc_n).sum()), vion + vh + vxc
    nd, vd = torch.tensor(n, device="cuda"), torch.empty(N, dtype=torch.float64, device="cuda")
    e = torch.zeros(2, dtype=torch.float64, device="cuda")
    jdft.jdft_hartree(b, nd, vd, e[:1])
    assert _rel(vd.cpu().numpy(), vh) < 64 * U64
    assert abs(float(e[0]) / eh - 1) < 64 * U64
    jdft.jdft_ks_potential(b, nd, torch.tensor(vion, device="cuda"), vd, e)
    assert _rel(vd.cpu().numpy(), vks) < 64 * U64
    assert abs(float(e[0]) / eh - 1) < 64 * U64 and abs(float(e[1]) / exc - 1) < 64 * U64


@pytest.mark.parametrize("S", RAGGED, ids=lambda s: "x".join(map(str, s)))
def test_ragged_lengths(S):
    """I, J and the Kohn-Sham potential on the other lengths.  Between passes the line of a large mean m keeps n m with a
    rounding of u n m, against sqrt(n) d for fluctuations d on it: the potential (no G = 0 term) of such a density is off by
    up to 8 u (1 + sqrt(n) m / d) in any FP64 transform."""
    jdft, b = _basis(S)
    N = int(np.prod(S))
    rng = np.random.default_rng(N + 2)
    x = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    xd = torch.tensor(x, device="cuda")
    out = torch.empty_like(xd)
    jdft.jdft_field_I(b, xd, out)
    assert _rel(out.cpu().numpy(), _I(S, x)) < 32 * U64
    jdft.jdft_field_J(b, xd, out)
    assert _rel(out.cpu().numpy(), _J(S, x)) < 32 * U64
    n = 0.05 * rng.random(N) + 1e-3
    vion = 0.1 * rng.standard_normal(N)
    K, nt, om = _coulomb(S), _J(S, n), LD(np.linalg.det(SKEW))
    vh = _I(S, K * nt).real
    eh = float(om / 2 * (K * np.abs(nt) ** 2).sum())
    exc_n, vxc = _lda(n)
    exc = float(om / N * (n * exc_n).sum())
    nd, vd = torch.tensor(n, device="cuda"), torch.empty(N, dtype=torch.float64, device="cuda")
    e = torch.zeros(2, dtype=torch.float64, device="cuda")
    tol = 8 * U64 * (1 + np.sqrt(max(S)) * n.mean() / n.std())
    jdft.jdft_hartree(b, nd, vd, e[:1])
    assert _rel(vd.cpu().numpy(), vh) < tol and abs(float(e[0]) / eh - 1) < 2 * tol
    jdft.jdft_ks_potential(b, nd, torch.tensor(vion, device="cuda"), vd, e)
    assert _rel(vd.cpu().numpy(), vion + vh + vxc) < tol
    assert abs(float(e[0]) / eh - 1) < 2 * tol and abs(float(e[1]) / exc - 1) < 64 * U64


@pytest.mark.parametrize("S", [BOXES[0], BOXES[3], BOXES[5], BOXES[7], BOXES[8], BOXES[9]] + RAGGED[::3],
                         ids=lambda s: "x".join(map(str, s)))
def test_dielectric_solve(S):
    """The hessian in FP64, and the FP32 solve, whose FP64 residual the library measures with it."""
    jdft, b = _basis(S)
    N = int(np.prod(S))
    rng = np.random.default_rng(N + 1)
    eps = 1.0 + 5.0 * rng.random(N)
    x = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    xd, ed, out = torch.tensor(x, device="cuda"), torch.tensor(eps, device="cuda"), torch.empty(
        N, dtype=torch.complex128, device="cuda")
    jdft.jdft_pcm_hessian(b, ed, xd, out)
    assert _rel(out.cpu().numpy(), _hessian(S, eps, x)) < 64 * U64
    x[0] = 0.0
    rep = jdft.jdft_pcm_solve(b, ed, torch.tensor(x, device="cuda"), out, tol=1e-11, prec="fp32")
    back = _hessian(S, eps, out.cpu().numpy())
    assert rep["residual"] <= 1e-11 and _rel(back, x) < 2e-11


def test_lda_points():
    jdft, b = _basis((12, 16, 40))
    N = 12 * 16 * 40
    n = 10.0 ** np.linspace(-35, 2, N - 40)
    n = np.concatenate([n, np.linspace(0.2290, 0.2400, 30), [0.0, -1e-3, 1e-30, 0.23, 1e-300, 5e-324, 1.0, 3.0, 7.0, 1e30]])
    v = torch.empty(N, dtype=torch.float64, device="cuda")
    nd = torch.tensor(n, device="cuda")
    jdft.jdft_xc_lda(b, nd, v)
    got = v.cpu().numpy()
    pos, ref = n > 0, _lda(n)[1]
    assert np.all(got[~pos] == 0.0)
    assert np.all(np.abs(got[pos] - ref[pos]) <= 16 * U64 * np.abs(ref[pos]))

"""The line-transform chain (line_path.cuh) on every compiled length along every axis, against numpy's long double.

H C without projectors, I, J and the density of FP64 and FP32 blocks.  Tolerances, relative to the result's norm (per
band): FP64 8 units of 2^-53 for H C and 6 for I and J (six and three line passes of at most a unit each and the products,
in quadrature, with a factor of two to spare; see test_gpu_fixfft.py); FP32 16 and 12 units of 2^-24, a pass being a
transform of up to eight FP32 roundings deep, two units; the density twice I's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [12, 16, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128,
           256]
BOXES = [(LENGTHS[i], LENGTHS[(i + 10) % 27], LENGTHS[(i + 19) % 27]) for i in range(27)]
UNIT = {"fp64": 2.0 ** -53, "fp32": 2.0 ** -24}
H_TOL, I_TOL = {"fp64": 8, "fp32": 16}, {"fp64": 6, "fp32": 12}


def _err(got, ref):
    d = np.abs(got - ref).reshape(len(ref), -1) ** 2
    return float(np.sqrt((d.sum(1) / (np.abs(ref) ** 2).reshape(len(ref), -1).sum(1)).max()))


@pytest.mark.parametrize("S", BOXES, ids=lambda s: "x".join(map(str, s)))
def test_chain(S, monkeypatch):
    import scipy.fft
    from paper_1708_03621_gb300 import jdft
    monkeypatch.setenv("JDFT_LINE_PATH", "1")
    ecut = 4.0
    L = [(s - 1.5) * 2 * np.pi / (4 * np.sqrt(2 * ecut)) for s in S]
    b = jdft.Basis(np.diag(L), S, ecut, [(0.1, 0.2, 0.3)])
    g = b.gvectors(0).astype(np.int64)
    npw, N, nb = len(g), int(np.prod(S)), 2
    q = (g + np.array([0.1, 0.2, 0.3])) * (2 * np.pi / np.array(L))
    rng = np.random.default_rng(N)
    C0 = (rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))) / (1 + (q * q).sum(1))
    V = -3.0 * rng.random(S) + 0.5
    psi0 = rng.standard_normal((nb, N)) + 1j * rng.standard_normal((nb, N))
    jdft.jdft_set_potential(b, torch.tensor(V.reshape(-1), device="cuda"))
    slot = ((g[:, 0] % S[0]) * S[1] + g[:, 1] % S[1]) * S[2] + g[:, 2] % S[2]
    T = (0.5 * (q * q).sum(1)).astype(np.longdouble)
    for prec, ct in (("fp64", np.complex128), ("fp32", np.complex64)):
        C, psi = C0.astype(ct), psi0.astype(ct)
        box = np.zeros((nb, N), dtype=np.clongdouble)
        box[:, slot] = C
        I = scipy.fft.ifftn(box.reshape((-1,) + S), axes=(1, 2, 3), norm="forward")
        back = scipy.fft.fftn(I * V.astype(np.longdouble), axes=(1, 2, 3), norm="forward").reshape(nb, -1)[:, slot]
        H = np.longdouble(np.prod(L)) * (T * C + back)
        J = scipy.fft.fftn(psi.astype(np.clongdouble).reshape((-1,) + S), axes=(1, 2, 3),
                           norm="forward").reshape(nb, -1)[:, slot]
        # a leading dimension past npw, which stays untouched
        Cd = torch.full((nb, npw + 3), 7.0, dtype=torch.complex128 if prec == "fp64" else torch.complex64, device="cuda")
        Cd[:, :npw] = torch.tensor(C, device="cuda")
        HC = torch.full_like(Cd, 5.0)
        jdft.jdft_profile_enable(True)
        jdft.jdft_profile_read()
        jdft.jdft_apply_H(b, 0, Cd, HC, prec=prec)
        torch.cuda.synchronize()
        names = jdft.jdft_profile_read()
        jdft.jdft_profile_enable(False)
        assert "line_columns" in names and "plane_apply" not in names
        u = UNIT[prec]
        assert _err(HC[:, :npw].cpu().numpy(), H) < H_TOL[prec] * u
        assert bool((HC[:, npw:] == 5.0).all())
        out = torch.empty((nb, N), dtype=Cd.dtype, device="cuda")
        jdft.jdft_op_I(b, 0, Cd, out, prec=prec)
        assert _err(out.cpu().numpy(), I.reshape(nb, -1)) < I_TOL[prec] * u
        back = torch.full_like(Cd, 5.0)
        jdft.jdft_op_J(b, 0, torch.tensor(psi, device="cuda"), back, prec=prec)
        assert _err(back[:, :npw].cpu().numpy(), J) < I_TOL[prec] * u
        f = torch.tensor([2.0, 0.7], dtype=torch.float64, device="cuda")
        n = torch.ones(N, dtype=torch.float64, device="cuda")
        jdft.jdft_density(b, 0, Cd, f, n, prec=prec)
        ref = 1.0 + 2.0 * np.abs(I[0]) ** 2 + 0.7 * np.abs(I[1]) ** 2
        assert _err(n.cpu().numpy()[None], ref.reshape(1, -1)) < 2 * I_TOL[prec] * u
        m = torch.zeros_like(n)
        jdft.jdft_apply_H_density(b, 0, Cd, HC, f, m, prec=prec)
        assert _err(HC[:, :npw].cpu().numpy(), H) < H_TOL[prec] * u
        assert _err(m.cpu().numpy()[None], ref.reshape(1, -1) - 1.0) < 2 * I_TOL[prec] * u

"""Performance cases of the plane-wave Hamiltonian library: the calls that programs built on it make, with their
inputs, one pass of each through the public binding, the work of a pass, and its result in 64 bits.

Cells, cutoffs, boxes, atoms and band counts are those of the repository's workloads (48^3 with 16 bands, 128^3 with
256 bands, the 256 x 128 x 128 slab with 1024 bands) and of its tests' box shapes, or the same recipe at other sizes:
Gaussian atoms at random positions with four projectors each, coefficients (x + iy) / (1 + |k+G|^2) with x, y standard
normal, k = (0.1, 0.2, 0.3).  Everything is drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1708_03621_gb300 import jdft

KFRAC = (0.1, 0.2, 0.3)
D_PER_ATOM = (0.5, -0.3, -0.3, -0.3)
#: Edges of the FFT boxes that cells are drawn on: the products of 2, 3 and 5 that the library takes, in the
#: range of the repository's workloads.
EDGES = (24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128)


# ---------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------
def _case(name, kind, S, L, ecut, atoms, bands, prec):
    return {"name": name, "kind": kind, "S0": S[0], "S1": S[1], "S2": S[2], "L0": L[0], "L1": L[1], "L2": L[2],
            "ecut": ecut, "atoms": atoms, "bands": bands, "prec": prec}


def listed():
    return [
        # H C on a molecule-sized cell in the binding's default precision: the inner call of a small
        # band solve, where launches and latency count.
        _case("apply_h_48_fp64", "apply_h", (48, 48, 48), (10.0,) * 3, 20.0, 8, 16, "fp64"),
        # The same call in the mixed precision: the smallest call of all.
        _case("apply_h_48_bf16x3", "apply_h", (48, 48, 48), (10.0,) * 3, 20.0, 8, 16, "bf16x3"),
        # An orthorhombic cell whose edges are no powers of two, an odd number of bands, plain FP32.
        _case("apply_h_ragged_fp32", "apply_h", (60, 54, 72), (13.9, 12.5, 16.5), 20.0, 11, 13, "fp32"),
        # A share of the large cell's bands in FP64: the finishing iterations of a large band solve.
        _case("apply_h_128_fp64", "apply_h", (128, 128, 128), (20.0,) * 3, 30.0, 64, 64, "fp64"),
        # One iteration's hot path on the large cell: H C, density, subspace matrices, orthonormalisation.
        _case("step_128_bf16x3", "step", (128, 128, 128), (20.0,) * 3, 30.0, 64, 256, "bf16x3"),
        # H C of the slab workload at one k-point: the largest block.
        _case("apply_h_slab_bf16x3", "apply_h", (256, 128, 128), (40.0, 20.0, 20.0), 30.0, 256, 1024, "bf16x3"),
        # The operators by themselves, as a program composes them (I, a pointwise product, J), on an odd box.
        _case("operators_ragged_fp64", "operators", (54, 60, 75), (12.5, 14.0, 17.5), 20.0, 9, 7, "fp64"),
        # Rayleigh-Ritz matrices and orthonormalisation of an FP64 block: once per outer iteration of a program
        # with its own minimiser.
        _case("subspace_80_fp64", "subspace", (80, 80, 80), (18.5,) * 3, 20.0, 20, 120, "fp64"),
        # A whole call: ten iterations of the band minimiser (one self-consistency step's band solve) in FP64.
        _case("minimize_48_fp64", "minimize", (48, 48, 48), (10.0,) * 3, 20.0, 8, 16, "fp64"),
        # Kohn-Sham potential of the large cell's density: once per self-consistency iteration.
        _case("ks_potential_128", "ks", (128, 128, 128), (20.0,) * 3, 30.0, 64, 256, "fp64"),
        # A whole call: the dielectric solve of the large cell's solute cavity, FP32 iterations with FP64 residuals.
        _case("pcm_solve_128_fp32", "pcm", (128, 128, 128), (20.0,) * 3, 30.0, 64, 0, "fp32"),
        # H C of spinor bands in a noncollinear potential on the large cell.
        _case("spinor_128_bf16x3", "spinor", (128, 128, 128), (20.0,) * 3, 30.0, 64, 64, "bf16x3"),
    ]


#: kind, weight, smallest and largest edge, largest band count and precisions of the drawn cases
_DRAWN = (
    ("apply_h", 5, 30, 128, 256, ("fp64", "fp64", "fp32", "tf32x3", "bf16x3")),
    ("operators", 2, 24, 96, 24, ("fp64", "fp32")),
    ("step", 2, 40, 128, 256, ("bf16x3",)),
    ("subspace", 2, 40, 108, 192, ("fp64", "fp64", "bf16x3")),
    ("minimize", 1, 30, 54, 24, ("fp64",)),
    ("ks", 2, 24, 128, 2, ("fp64",)),
    ("pcm", 1, 30, 128, 2, ("fp32", "fp64")),
    ("spinor", 1, 30, 128, 64, ("fp64", "fp32", "bf16x3")),
)


def draw(rng):
    """A case of the ranges above: edges spread over their logarithm (a third of the cells cubic), the cell as large
    as the box holds at the cutoff, band counts over their logarithm (FP64 blocks up to a quarter of the largest)."""
    kind, _, lo, hi, most, precs = rng.choices(_DRAWN, weights=[d[1] for d in _DRAWN])[0]
    prec = rng.choice(precs)
    ecut = rng.choice((12.0, 20.0, 30.0))

    def edge():
        x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min((e for e in EDGES if lo <= e <= hi), key=lambda e: abs(e - x))

    S = (edge(),) * 3 if rng.random() < 0.34 else (edge(), edge(), edge())
    # twice the sphere's reach fits the box: 4 sqrt(2 E) L / 2 pi + 1 <= S
    L = [round((s - 1.5) * 2.0 * math.pi / (4.0 * math.sqrt(2.0 * ecut)), 3) for s in S]
    npw = L[0] * L[1] * L[2] * (2.0 * ecut) ** 1.5 / (6.0 * math.pi ** 2)
    if prec == "fp64":
        most = max(2, most // 4) if kind in ("apply_h", "spinor") else most
    most = max(1, min(most, int(npw / 24)))
    bands = int(round(math.exp(rng.uniform(0.0, math.log(most))))) if most > 1 else 1
    if kind in ("step", "subspace", "minimize"):
        bands = max(4, bands)
    atoms = max(1, min(64, int(rng.uniform(0.5, 1.2) * 8.0 * L[0] * L[1] * L[2] / 1000.0)))
    c = _case("", kind, S, L, ecut, atoms, 0 if kind == "pcm" else bands, prec)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _box(case):
    S = (case["S0"], case["S1"], case["S2"])
    L = torch.tensor([case["L0"], case["L1"], case["L2"]], dtype=torch.float64, device="cuda")
    return S, L, S[0] * S[1] * S[2], float(case["L0"] * case["L1"] * case["L2"])


def _rng(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + salt)
    return g


def _atoms(case, seed):
    _, L, _, _ = _box(case)
    return torch.rand((case["atoms"], 3), generator=_rng(seed, 0), dtype=torch.float64, device="cuda") * L


def _gaussians(case, centres, width, weights=None):
    """sum_a w_a sum over images of exp(-|r - R_a|^2 / 2 width^2) on the box (orthorhombic cells: separable)."""
    S, L, _, _ = _box(case)
    ax = []
    for d in range(3):
        x = L[d] * torch.arange(S[d], dtype=torch.float64, device="cuda") / S[d]
        reach = int(math.ceil(10.0 * width / float(L[d]))) + 1
        im = torch.arange(-reach, reach + 1, dtype=torch.float64, device="cuda") * L[d]
        dx = x[None, :, None] - centres[:, d, None, None] - im[None, None, :]
        ax.append(torch.exp(-0.5 * (dx / width) ** 2).sum(-1))
    if weights is not None:
        ax[0] = ax[0] * weights[:, None]
    xy = (ax[0][:, :, None] * ax[1][:, None, :]).reshape(len(centres), -1)
    return (xy.T @ ax[2]).reshape(-1)


def _sphere(case):
    """Integer triples of the plane-wave sphere in lexicographic order (npw x 3) and Cartesian k+G."""
    kmax = math.sqrt(2.0 * case["ecut"])
    ax = []
    for d in range(3):
        reach = int(math.ceil(case["L%d" % d] * kmax / (2.0 * math.pi))) + 2
        ax.append(torch.arange(-reach, reach + 1, device="cuda"))
    g = torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)
    _, L, _, _ = _box(case)
    q = (g + torch.tensor(KFRAC, dtype=torch.float64, device="cuda")) * (2.0 * math.pi / L)
    keep = 0.5 * (q * q).sum(-1) <= case["ecut"]
    return g[keep], q[keep]


def _block(case, q, rows, seed, salt=1):
    """Band-major coefficient block: (x + iy) / (1 + |k+G|^2), in the precision's block type."""
    t = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    r = torch.float64 if case["prec"] == "fp64" else torch.float32
    C = torch.randn((rows, q.shape[0], 2), generator=_rng(seed, salt), dtype=r, device="cuda")
    C /= (1.0 + (q * q).sum(-1)).to(r)[None, :, None]
    return torch.view_as_complex(C).to(t)


def _projectors(case, q, atoms):
    """P (4 atoms x npw, projector-major) of unit-width Gaussian s and p functions, and the diagonal D."""
    q2 = (q * q).sum(-1)
    Ns = math.pi ** -0.75
    Fs = Ns * (2.0 * math.pi) ** 1.5 * torch.exp(-0.5 * q2)
    F = torch.stack([Fs.to(torch.complex128)] + [-1j * math.sqrt(2.0) * q[:, d] * Fs for d in range(3)])
    ph = atoms @ q.T
    P = torch.empty((atoms.shape[0], 4, q.shape[0]), dtype=torch.complex128, device="cuda")
    torch.mul(torch.polar(torch.ones_like(ph), -ph)[:, None, :], F[None], out=P)
    D = torch.diag(torch.tensor(D_PER_ATOM * atoms.shape[0], dtype=torch.float64, device="cuda"))
    return P.reshape(-1, q.shape[0]), D


def _density(case, seed):
    """A positive density: the atoms' Gaussians on a rippled background."""
    S, L, N, _ = _box(case)
    n = 0.08 * _gaussians(case, _atoms(case, seed), 1.1)
    ripple = torch.rand(N, generator=_rng(seed, 5), dtype=torch.float64, device="cuda")
    return n + 2e-3 * (0.5 + ripple)


def _cavity(case, seed):
    """eps(r) of a smooth solute cavity (1 inside, 78.4 far away) and rho~ of charges at its centres."""
    S, L, N, omega = _box(case)
    at = _atoms(case, seed)
    q = torch.randn(case["atoms"], generator=_rng(seed, 6), dtype=torch.float64, device="cuda")
    eps = 1.0 + 77.4 * torch.exp(-6.0 * _gaussians(case, at, 2.0))
    rho = _gaussians(case, at, 1.0, q - q.mean())
    return eps, torch.fft.fftn(rho.reshape(S).to(torch.complex128), norm="forward").reshape(-1).contiguous()


def _field(case, seed):
    """A noncollinear field M (3 N): Gaussians at random points, another set for each component."""
    S, L, N, _ = _box(case)
    M = []
    for c in range(3):
        at = torch.rand((6, 3), generator=_rng(seed, 7 + c), dtype=torch.float64, device="cuda") * L
        M.append(0.3 * _gaussians(case, at, 1.5) - 0.1)
    return torch.cat(M).contiguous()


def _basis(case):
    S, _, _, _ = _box(case)
    return jdft.Basis(np.diag([case["L0"], case["L1"], case["L2"]]), S, case["ecut"], [KFRAC])


def _inputs(case, seed):
    """The plain tensors a case starts from, the same for run() and exact()."""
    kind = case["kind"]
    if kind == "ks":
        return {"n": _density(case, seed), "vion": -4.0 * _gaussians(case, _atoms(case, seed), 1.0)}
    if kind == "pcm":
        eps, rho = _cavity(case, seed)
        return {"eps": eps, "rho": rho}
    _, q = _sphere(case)
    s = {"C": _block(case, q, case["bands"] * (2 if kind == "spinor" else 1), seed)}
    if kind == "subspace":
        s["HC"] = _block(case, q, case["bands"], seed, 2) + (0.5 * (q * q).sum(-1)).to(s["C"].dtype) * s["C"]
        return s
    at = _atoms(case, seed)
    s["V"] = -4.0 * _gaussians(case, at, 1.0)
    if kind == "operators":
        return s
    s["P"], s["D"] = _projectors(case, q, at)
    if kind == "spinor":
        s["M"] = _field(case, seed)
    if kind == "step":
        s["f"] = torch.full((case["bands"],), 2.0, dtype=torch.float64, device="cuda")
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"], s["prec"], s["basis"] = case["kind"], case["prec"], _basis(case)
    b, nb, N = s["basis"], case["bands"], _box(case)[2]
    real, cplx = {"dtype": torch.float64, "device": "cuda"}, {"dtype": torch.complex128, "device": "cuda"}
    if "V" in s and case["kind"] != "operators":
        jdft.jdft_set_potential(b, s.pop("V"))
    if "P" in s:
        jdft.jdft_set_projectors(b, 0, s.pop("P"), s.pop("D"))
    if case["kind"] in ("apply_h", "spinor", "step"):
        s["HC"] = torch.empty_like(s["C"])
    if case["kind"] in ("step", "subspace"):
        s["CHC"], s["COC"] = torch.empty((nb, nb), **cplx), torch.empty((nb, nb), **cplx)
    if case["kind"] == "step":
        s["n"], s["status"] = torch.empty(N, **real), torch.zeros(1, dtype=torch.int32, device="cuda")
    if case["kind"] == "operators":
        s["psi"] = torch.empty((nb,) + _box(case)[0], dtype=s["C"].dtype, device="cuda")
        s["V"] = s["V"].reshape(_box(case)[0]).to(s["psi"].real.dtype)
        s["out"] = torch.empty_like(s["C"])
    if case["kind"] == "minimize":
        s["start"], s["eigs"] = s["C"].clone(), torch.empty(nb, **real)
    if case["kind"] == "ks":
        s["vks"], s["energies"] = torch.empty(N, **real), torch.empty(2, **real)
    if case["kind"] == "pcm":
        s["phi"] = torch.empty(N, **cplx)
    return s


# ---------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------
def run(s):
    b, kind, prec = s["basis"], s["kind"], s["prec"]
    if kind == "apply_h":
        jdft.jdft_apply_H(b, 0, s["C"], s["HC"], prec=prec)
        return s["HC"]
    if kind == "spinor":
        jdft.jdft_apply_H_spinor(b, 0, s["M"], s["C"], s["HC"], prec=prec)
        return s["HC"]
    if kind == "operators":
        jdft.jdft_op_I(b, 0, s["C"], s["psi"], prec=prec)
        phi = s["psi"] * s["V"]
        jdft.jdft_op_J(b, 0, phi, s["out"], prec=prec)
        return s["psi"], s["out"]
    if kind == "step":
        s["n"].zero_()
        jdft.jdft_hamiltonian_step(b, 0, s["C"], s["HC"], s["f"], s["n"], s["CHC"], s["COC"], s["status"], prec=prec)
        # the mixed path's density and subspace matrices hold single-precision results in FP64 containers;
        # a mixed program goes on with them in the type of its blocks
        return s["HC"], s["C"], s["n"].float(), s["CHC"].to(s["C"].dtype), s["COC"].to(s["C"].dtype)
    if kind == "subspace":
        jdft.jdft_subspace(b, 0, s["C"], s["HC"], s["CHC"], s["COC"], prec=prec)
        jdft.jdft_orthonormalize(b, 0, s["C"], prec=prec)
        return s["C"], s["CHC"].to(s["C"].dtype), s["COC"].to(s["C"].dtype)
    if kind == "minimize":
        s["C"].copy_(s["start"])
        r = jdft.jdft_minimize_bands(b, 0, s["C"], eigs=s["eigs"], tol=1e-12, max_iter=10, prec=prec, check=False)
        return s["C"], s["eigs"], r["energy"], r["iterations"]
    if kind == "ks":
        jdft.jdft_ks_potential(b, s["n"], s["vion"], s["vks"], s["energies"])
        return s["vks"], s["energies"]
    r = jdft.jdft_pcm_solve(b, s["eps"], s["rho"], s["phi"], tol=1e-11, prec=prec)
    return s["phi"], r["A_diel"]


# ---------------------------------------------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------------------------------------------
def work(case):
    """Inputs read once, outputs written once; transforms counted as 5 n log2 n per line, of the lines that the
    sphere touches, products as 8 per complex multiply-add."""
    S, _, N, omega = _box(case)
    kind, nb = case["kind"], case["bands"]
    kmax = math.sqrt(2.0 * case["ecut"])
    npw = omega * kmax ** 3 / (6.0 * math.pi ** 2)
    cols = case["L0"] * case["L1"] * kmax ** 2 / (4.0 * math.pi)
    rows = min(S[0], case["L0"] * kmax / math.pi)
    line = [5.0 * n * math.log2(n) for n in S]
    box = sum(line[d] * N / S[d] for d in range(3))
    sphere = cols * line[2] + rows * S[2] * line[1] + S[1] * S[2] * line[0]
    nproj, w = 4 * case["atoms"], 16.0 if case["prec"] == "fp64" else 8.0
    if kind in ("apply_h", "spinor", "step"):
        r = nb * (2 if kind == "spinor" else 1)
        out = {"bytes": 2 * r * npw * w + nproj * npw * w + 8.0 * N * (4 if kind == "spinor" else 1),
               "flops": r * 2 * sphere + 16.0 * nproj * r * npw}
        if kind == "step":
            out = {"bytes": out["bytes"] + nb * npw * w + 8.0 * N + 32.0 * nb * nb,
                   "flops": out["flops"] + 8.0 * npw * nb * nb * (0.5 + 0.5 + 0.5)}
        return out
    if kind == "operators":
        return {"bytes": nb * w * (2 * npw + 2 * N) + 0.5 * w * N, "flops": nb * (2 * sphere + 2 * N)}
    if kind == "subspace":
        return {"bytes": 3 * nb * npw * w + 32.0 * nb * nb, "flops": 8.0 * npw * nb * nb * (1 + 0.5 + 0.5)}
    if kind == "minimize":
        # per iteration one H C, the projection and rotation products, the block read and written
        return {"bytes": 10 * (4 * nb * npw * w + nproj * npw * w + 8.0 * N),
                "flops": 10 * (nb * 2 * sphere + 16.0 * nproj * nb * npw + 4 * 8.0 * npw * nb * nb)}
    if kind == "ks":
        return {"bytes": 24.0 * N, "flops": box + 100.0 * N}  # two transforms of real fields
    # about a hundred iterations (a hundredfold dielectric), six transforms each
    return {"bytes": 40.0 * N, "flops": 100 * 6 * box}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------------------------
def _slots(g, S):
    return ((g[:, 0] % S[0]) * S[1] + g[:, 1] % S[1]) * S[2] + g[:, 2] % S[2]


def _I(C, slots, S):
    box = torch.zeros((C.shape[0], S[0] * S[1] * S[2]), dtype=torch.complex128, device="cuda")
    box[:, slots] = C
    return torch.fft.ifftn(box.reshape((-1,) + S), dim=(1, 2, 3), norm="forward")


def _J(x, slots, S):
    return torch.fft.fftn(x.reshape((-1,) + S), dim=(1, 2, 3), norm="forward").reshape(x.shape[0], -1)[:, slots]


def _local(C, V, slots, S, M=None, n=None):
    """J (V I C) by groups of bands, for spinor rows with V + M . sigma; adds 2 |I C|^2 to n."""
    out = torch.empty_like(C)
    V = V.reshape(S)
    step = max(2, min(64, int(2e8 // V.numel()) // 2 * 2))
    for a in range(0, C.shape[0], step):
        psi = _I(C[a:a + step], slots, S)
        if n is not None:
            n += 2.0 * (psi.real ** 2 + psi.imag ** 2).sum(0).reshape(-1)
        if M is None:
            psi *= V
        else:
            mx, my, mz = M.reshape((3,) + S)
            up, dn = psi[0::2], psi[1::2]
            psi = torch.stack([(V + mz) * up + (mx - 1j * my) * dn, (mx + 1j * my) * up + (V - mz) * dn],
                              dim=1).reshape(psi.shape)
        out[a:a + step] = _J(psi, slots, S)
    return out


def _lda(n):
    """e_xc and v_xc per point: Slater exchange and the Perdew-Zunger fit of correlation (n > 0)."""
    ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * n ** (1.0 / 3.0)
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    sq, lr = rs.sqrt(), rs.log()
    den = 1.0 + 1.0529 * sq + 0.3334 * rs
    ec = torch.where(rs >= 1.0, -0.1423 / den, 0.0311 * lr - 0.048 + 0.002 * rs * lr - 0.0116 * rs)
    dec = torch.where(rs >= 1.0, 0.1423 * (0.5 * 1.0529 / sq + 0.3334) / den ** 2,
                      0.0311 / rs + 0.002 * (lr + 1.0) - 0.0116)
    return ex + ec, 4.0 / 3.0 * ex + ec - rs / 3.0 * dec


def _box_G(case):
    S, L, _, _ = _box(case)
    ax = [torch.fft.fftfreq(S[d], 1.0 / S[d], dtype=torch.float64, device="cuda").round() * (2 * math.pi / L[d])
          for d in range(3)]
    return torch.meshgrid(*ax, indexing="ij")


def _coulomb(case):
    G2 = sum(g * g for g in _box_G(case))
    return torch.where(G2 > 0, 4.0 * math.pi / torch.where(G2 > 0, G2, 1.0), 0.0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "minimize":
        return None
    s = _inputs(case, seed)
    S, _, N, omega = _box(case)
    if kind == "ks":
        n, K = s["n"], _coulomb(case)
        nt = torch.fft.fftn(n.reshape(S).to(torch.complex128), norm="forward")
        vh = torch.fft.ifftn(K * nt, norm="forward").real.reshape(-1)
        e, v = _lda(n)
        eh = 0.5 * omega * (K * (nt.real ** 2 + nt.imag ** 2)).sum()
        return s["vion"] + vh + v, torch.stack([eh, omega / N * (n * e).sum()])
    if kind == "pcm":
        return _exact_pcm(case, s["eps"].reshape(S), s["rho"].reshape(S))
    C = s["C"].to(torch.complex128)
    if kind == "subspace":
        CHC, COC = C.conj() @ s["HC"].to(torch.complex128).T, omega * (C.conj() @ C.T)
        return _orthonormal(C, COC), CHC, COC
    g, q = _sphere(case)
    slots = _slots(g, S)
    if kind == "operators":
        psi = _I(C, slots, S)
        return psi, _J(psi * s["V"].reshape(S), slots, S)
    n = torch.zeros(N, dtype=torch.float64, device="cuda") if kind == "step" else None
    HC = _local(C, s["V"], slots, S, s.get("M"), n)
    HC += (0.5 * (q * q).sum(-1)) * C
    HC *= omega
    HC += ((s["P"].conj() @ C.T) * torch.diagonal(s["D"])[:, None]).T @ s["P"]
    if kind != "step":
        return HC
    CHC, COC = C.conj() @ HC.T, omega * (C.conj() @ C.T)
    return HC, _orthonormal(C, COC), n, CHC, COC


def _orthonormal(C, COC):
    """C L^{-dag} with COC = L L^dag, for a band-major block."""
    return torch.linalg.solve_triangular(torch.linalg.cholesky(COC).conj(), C, upper=False)


def _exact_pcm(case, eps, rho):
    G, K = _box_G(case), _coulomb(case)
    _, _, _, omega = _box(case)
    rho = torch.where(K > 0, rho, 0.0)

    def hessian(x):
        out = 0
        for d in range(3):
            out = out + 1j * G[d] * torch.fft.fftn(eps * torch.fft.ifftn(1j * G[d] * x, norm="forward"),
                                                   norm="forward")
        return out / (-4.0 * math.pi)

    def dot(a, b):
        return (a.real * b.real + a.imag * b.imag).sum()

    x, r = torch.zeros_like(rho), rho.clone()
    z = K * r
    d, rz, want = z.clone(), dot(r, z), 1e-14 * torch.sqrt(dot(rho, rho))
    for _ in range(250):
        Hd = hessian(d)
        a = rz / dot(d, Hd)
        x, r = x + a * d, r - a * Hd
        if torch.sqrt(dot(r, r)) < want:
            break
        z = K * r
        new = dot(r, z)
        d, rz = z + new / rz * d, new
    return x.reshape(-1), 0.5 * omega * dot(x - K * rho, rho)

"""The sliced FP64 products (tc_slices.cuh) when their bounded waits run out: the limit at 0 makes each give up at its
first wait.  A product that gave up says so in its output (NaN, never a sum of what the scratch held before), in
jdft_device_status, and in the return value of a call that waits for it; the next call gives the same bits as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NB = 64


def _system():
    from paper_1708_03621_gb300 import jdft
    b = jdft.Basis(np.eye(3) * 10.0, (48, 48, 48), 20.0, [(0.1, 0.2, 0.3)])
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    C = torch.view_as_complex(torch.randn((NB, b.npw(0), 2), generator=g, dtype=torch.float64, device="cuda"))
    V = torch.rand(48 ** 3, generator=g, dtype=torch.float64, device="cuda")
    jdft.jdft_set_potential(b, V)
    P = torch.view_as_complex(torch.randn((128, b.npw(0), 2), generator=g, dtype=torch.float64, device="cuda")) * 1e-3
    jdft.jdft_set_projectors(b, 0, P, torch.eye(128, dtype=torch.float64, device="cuda"))
    return jdft, b, C


def _timed_out(jdft, call):
    jdft.jdft_set_wait_limit(0.0)
    try:
        with pytest.raises(jdft.JdftError) as err:
            call()
        assert err.value.status == jdft.STATUS_CODES["ERR_TIMEOUT"]
    finally:
        jdft.jdft_set_wait_limit(2.0)


def test_products_that_give_up_are_nan_and_the_next_are_whole():
    jdft, b, C = _system()
    H = C.flip(0).contiguous()
    ref, got = (torch.empty((2, NB, NB), dtype=torch.complex128, device="cuda") for _ in range(2))
    hc = torch.empty_like(C)
    jdft.jdft_subspace(b, 0, C, H, ref[0], ref[1])
    jdft.jdft_apply_H(b, 0, C, hc)
    jdft.jdft_device_status()

    def call():
        jdft.jdft_subspace(b, 0, C, H, got[0], got[1])
        jdft.jdft_apply_H(b, 0, C, out)
        jdft.jdft_device_status()

    out = torch.empty_like(C)
    _timed_out(jdft, call)
    assert torch.isnan(got.real).all() and torch.isnan(got.imag).all()
    assert torch.isnan(out.real).all() and torch.isnan(out.imag).all()
    jdft.jdft_device_status()  # read and cleared
    jdft.jdft_subspace(b, 0, C, H, got[0], got[1])
    jdft.jdft_apply_H(b, 0, C, out)
    jdft.jdft_device_status()
    assert torch.equal(got, ref) and torch.equal(out, hc)


@pytest.mark.parametrize("name", ["orthonormalize", "minimize", "orthonormalize_generalized", "subspace_generalized",
                                  "subspace_generalized_without_eigenvalues", "minimize_generalized", "mlp_rows"])
def test_calls_that_wait_return_the_timeout(name):
    jdft, b, C = _system()
    if "generalized" in name:
        jdft.jdft_set_augmentation(b, 0, 1e-2 * torch.eye(128, dtype=torch.float64, device="cuda"))
    S = torch.empty((2, NB, NB), dtype=torch.complex128, device="cuda")
    eigs = torch.empty(NB, dtype=torch.float64, device="cuda")
    calls = {
        "orthonormalize": lambda D: jdft.jdft_orthonormalize(b, 0, D),
        "minimize": lambda D: jdft.jdft_minimize_bands(b, 0, D, tol=1e-9, max_iter=2),
        "orthonormalize_generalized": lambda D: jdft.jdft_orthonormalize_generalized(b, 0, D),
        "subspace_generalized": lambda D: jdft.jdft_subspace_generalized(b, 0, D, C, S[0], S[1], eigs),
        "subspace_generalized_without_eigenvalues":
            lambda D: jdft.jdft_subspace_generalized(b, 0, D, C, S[0], S[1], None),
        "mlp_rows": lambda D: jdft.jdft_mlp_rows(b, 0, D, C),
        "minimize_generalized": lambda D: jdft.jdft_minimize_bands_generalized(b, 0, D, tol=1e-9, max_iter=2),
    }
    _timed_out(jdft, lambda: calls[name](C.clone()))
    with pytest.raises(jdft.JdftError):
        jdft.jdft_device_status()
    # the failure is not remembered against the next call
    D = C.clone()
    jdft.jdft_orthonormalize(b, 0, D)
    eye = 1000.0 * (D.conj() @ D.T)
    assert float((eye - torch.eye(NB, device="cuda")).abs().max()) < 1e-12

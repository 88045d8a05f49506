"""jdft_subspace_eigs of graded matrices: cyclic Jacobi keeps the relative accuracy of decoupled small blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, scale", [(5, 1e-20), (6, 1e-20), (20, 1e-25), (61, 1e-30), (70, 1e-22)])
def test_small_block_beside_a_large_diagonal(n, scale):
    """Eigenvalues of diag(1, 2, 3) + scale x (random n x n): those of the small block by themselves, within the n units
    of 2^-53 of its norm that a sweep may cost, some ten sweeps: 16 n units, both sides."""
    from paper_1708_03621_gb300 import jdft
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    B = B + B.conj().T
    A = np.zeros((n + 3, n + 3), dtype=np.complex128)
    A[:3, :3] = np.diag([1.0, 2.0, 3.0])
    A[3:, 3:] = scale * B
    e = torch.empty(n + 3, dtype=torch.float64, device="cuda")
    jdft.jdft_subspace_eigs(torch.tensor(A, device="cuda"), e)
    got = e.cpu().numpy()
    ref = np.linalg.eigvalsh(B)
    assert np.array_equal(got[-3:], [1.0, 2.0, 3.0])
    assert np.abs(got[:n] / scale - ref).max() <= 16 * n * 2.0 ** -53 * np.abs(ref).max()

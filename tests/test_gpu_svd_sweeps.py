"""The sweep count of the Jacobi SVD: sweeps that rotated, also where every
rotation of the last one was too small to ask for another."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [24, 40, 101])  # one cluster, the whole GPU, an odd count
def test_a_sweep_of_small_rotations_counts(n):
    """Columns of distinct norms with cosines of about 1e-12, above the threshold
    (3.6e-15) and below what asks for another sweep (1e-10): one sweep."""
    import torch
    import paper_2603_17711_gb300 as pkg
    rng = np.random.default_rng(n)
    g = lambda *s: rng.normal(size=s) + 1j * rng.normal(size=s)  # noqa: E731
    q = np.linalg.qr(g(2 * n, n))[0] * np.linspace(1.0, 2.0, n)
    a = q + 1e-12 * g(2 * n, n) / np.sqrt(2 * n)
    U, s, Vh, sweeps = pkg.svd(torch.as_tensor(a, device="cuda"))
    assert sweeps == 1
    assert pkg.svd(torch.as_tensor(np.eye(2 * n, n, dtype=np.complex128), device="cuda"))[3] == 0
    u = U.cpu().numpy()
    assert np.max(np.abs(u.conj().T @ u - np.eye(n))) <= 1e-13

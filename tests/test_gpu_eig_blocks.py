"""Clusters of eigenvalues that belong to different blocks of the tridiagonal form.

A matrix of two diagonal blocks whose eigenvalues differ by `shift` falls apart in the reduction;
the pairs are closer than the direct path tells apart, and each vector must come with the eigenvalue
of its own block, in ascending order, whichever block comes first.  Tolerance as in test_gpu_eig.py,
with no allowance for the width of a cluster: n 2^-52 ||A||."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


def two_blocks(h, shift, seed):
    rng = np.random.default_rng(seed)
    A = np.zeros((2 * h, 2 * h))
    for b in range(2):
        Q, _ = np.linalg.qr(rng.standard_normal((h, h)))
        B = (Q * (np.linspace(-1.0, 1.0, h) + b * shift)) @ Q.T
        A[b * h:(b + 1) * h, b * h:(b + 1) * h] = 0.5 * (B + B.T)
    return A


@pytest.mark.parametrize("shift", [-2.0 ** -44, 2.0 ** -44, -2.0 ** -48, 2.0 ** -47])
@pytest.mark.parametrize("h,k", [(15, 30), (30, 60), (30, 21), (80, 40), (80, 160), (200, 45)])
def test_each_vector_has_the_eigenvalue_of_its_block(h, k, shift):
    A, n = two_blocks(h, shift, h), 2 * h
    w, Z = dfscf.eigh_lowest(A, k) if k < n else dfscf.eigh(A)
    w, Z = w.cpu().numpy(), Z.cpu().numpy()
    tol = n * 2.0 ** -52
    assert np.all(np.diff(w) >= 0.0)
    assert np.max(np.abs(w - np.linalg.eigvalsh(A)[:k])) <= tol
    assert np.max(np.abs(Z.T @ Z - np.eye(k))) <= tol
    assert np.max(np.abs(A @ Z - Z * w)) <= tol


@pytest.mark.parametrize("n", [40, 200])
def test_many_small_blocks(n):
    """Eigenvalues 2^-46 apart, in descending order along the diagonal: n blocks of one row."""
    d = 1.0 - 2.0 ** -46 * np.arange(n)
    w, Z = dfscf.eigh(np.diag(d))
    w, Z = w.cpu().numpy(), Z.cpu().numpy()
    assert np.max(np.abs(w - d[::-1])) <= 2.0 ** -52
    assert np.max(np.abs(Z.T @ Z - np.eye(n))) <= 2.0 ** -52
    assert np.max(np.abs(d[:, None] * Z - Z * w)) <= 2.0 ** -51

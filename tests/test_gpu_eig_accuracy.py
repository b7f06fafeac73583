"""Eigenvectors of a tridiagonal matrix, to the rounding of their elements.

The reduction leaves a tridiagonal matrix as it is, so what is tested is the direct vectors: a
factorisation in FP64 alone leaves components of size 2^-53 ||T|| / gap along the neighbours
(1e-14 here), and the correction with the residual in twice the precision has to remove them.
What remains is the rounding of z, of its norm and of the re-orthonormalisation: 8 units of 2^-53.

Reference: Rayleigh quotient iteration on the pivots of both factorisations in numpy's long double."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
LD = np.longdouble


def reference(d, e, w):
    """Unit eigenvector next to w in long double."""
    n = len(d)
    d, e = d.astype(LD), e.astype(LD)
    l = LD(w)
    for _ in range(4):
        q, p = np.empty(n, LD), np.empty(n, LD)
        q[0], p[n - 1] = d[0] - l, d[n - 1] - l
        for i in range(1, n):
            q[i] = d[i] - l - e[i - 1] ** 2 / q[i - 1]
        for i in range(n - 2, -1, -1):
            p[i] = d[i] - l - e[i] ** 2 / p[i + 1]
        r = int(np.argmin(np.abs(q + p - (d - l))))
        z = np.zeros(n, LD)
        z[r] = 1
        for i in range(r - 1, -1, -1):
            z[i] = -e[i] / q[i] * z[i + 1]
        for i in range(r + 1, n):
            z[i] = -e[i - 1] / p[i] * z[i - 1]
        z /= np.sqrt((z * z).sum())
        l = (d * z * z).sum() + 2 * (e * z[1:] * z[:-1]).sum()
    return z


@pytest.mark.parametrize("n,k,seed", [(9, 3, 0), (64, 9, 1), (150, 30, 2), (301, 20, 3)])
def test_vectors_of_a_tridiagonal_matrix(n, k, seed):
    rng = np.random.default_rng(seed)
    d = rng.standard_normal(n)
    e = np.sqrt(rng.chisquare(np.arange(n - 1, 0, -1)) / n)  # as the reduction of a random matrix leaves it
    A = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    w, Z = dfscf.eigh_lowest(A, k)
    w, Z = w.cpu().numpy(), Z.cpu().numpy()
    assert np.min(np.diff(w)) > 1e-4
    for t in range(k):
        z = reference(d, e, w[t])
        v = Z[:, t] * np.sign(float(z @ Z[:, t]))
        assert float(np.max(np.abs(v - z))) <= 8 * 2.0 ** -53

"""What the direct eigenvectors leave to their fallbacks.

A dense matrix with a cluster of m eigenvalues closer than the direct path tells apart stays one
block of its tridiagonal form; with m n > 4096 the CTAs of that cluster hand the solve over while
other CTAs of the same launch are still starting (at 900 rows they come in several waves).  The
hand-over is asserted from the solve's control record in the workspace, found by a poll limit
that only this test sets.

Tolerance: as in test_gpu_eig.py, n 2^-52 ||A|| for eigenvalues and orthonormality.  Vectors of a
cluster may be any basis of its space, so their residual may reach the cluster's width."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
POLLS = 4194301


def clustered(n, m, gap, seed):
    """(A, eigenvalues): the lowest m eigenvalues `gap` apart, the others spread up to 1."""
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    w = np.concatenate([-1.0 + gap * np.arange(m), np.linspace(-0.5, 1.0, n - m)])
    A = (Q * w) @ Q.T
    return 0.5 * (A + A.T), w


def solve(A, k):
    """Eigenpairs, whether the direct vectors were given up, and whether they were made at all."""
    lib, n = dfscf.lib(), len(A)
    dev = torch.as_tensor(A, device="cuda").clone()
    w = torch.empty(k, dtype=torch.float64, device="cuda")
    Z = torch.empty(n, k, dtype=torch.float64, device="cuda")
    need = lib.df_eigh_work_bytes(n) if k == n else lib.df_eigh_lowest_work_bytes(n, k)
    work = torch.zeros((need + 1023) // 1024 * 1024, dtype=torch.uint8, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (dev, w, Z, work)]
    old = lib.df_tune_get(b"eig_barrier_polls")
    lib.df_tune_set(b"eig_barrier_polls", POLLS)
    try:
        if k == n:
            rc = lib.df_eigh(ptr[0], n, ptr[1], ptr[2], ptr[3], work.numel(), None)
        else:
            rc = lib.df_eigh_lowest(ptr[0], n, k, ptr[1], ptr[2], ptr[3], work.numel(), None)
    finally:
        lib.df_tune_set(b"eig_barrier_polls", old)
    assert rc == dfscf.DF_OK, lib.df_last_error()
    words = work.view(torch.int32)[-1024:].cpu().numpy()
    at = np.flatnonzero(words == POLLS)
    assert len(at) == 1
    return w.cpu().numpy(), Z.cpu().numpy(), bool(words[at[0] + 1]), bool(words[at[0] + 3:at[0] + 5].any())


@pytest.mark.parametrize("n,m,k,direct", [(120, 20, 60, True), (120, 40, 60, False), (120, 40, 120, False),
                                          (300, 30, 40, False), (900, 400, 900, False)])
def test_clusters_beyond_the_direct_path(n, m, k, direct):
    gap = 2.0 ** -44
    A, ref = clustered(n, m, gap, n + m)
    w, Z, gave_up, _ = solve(A, k)
    assert gave_up != direct
    tol = n * 2.0 ** -52
    assert np.max(np.abs(w - ref[:k])) <= tol
    assert np.max(np.abs(Z.T @ Z - np.eye(k))) <= tol
    R = np.abs(A @ Z - Z * w)
    assert np.max(R[:, m:k]) <= tol
    assert np.max(R[:, :m]) <= tol + m * gap


@pytest.mark.parametrize("n", [1704, 1705, 1814, 1815])
def test_largest_rows_in_shared_memory(n):
    """Up to 1814 rows (152 SMs) the reduction keeps its rows in shared memory, from 1705 on with
    one vector less; beyond, the general path takes over."""
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 40))
    A = X @ X.T / n + np.diag(np.linspace(-1.0, 1.0, n))
    A = 0.5 * (A + A.T)
    w, Z, gave_up, direct = solve(A, 30)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert direct == (n <= 1814) and not gave_up
    ref = np.linalg.eigvalsh(A)
    tol, norm = n * 2.0 ** -52, np.max(np.abs(ref))
    assert np.max(np.abs(w - ref[:30])) <= tol * norm
    assert np.max(np.abs(Z.T @ Z - np.eye(30))) <= tol
    assert np.max(np.abs(A @ Z - Z * w)) <= tol * norm

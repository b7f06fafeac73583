"""The multi-SM eigensolver at the edges of its tiles: column counts around 128 (one column per
thread), 256, 512 and 1024, panels of 16 reflectors, minors in blocks of 8, row counts per CTA that
are not a multiple of 8, and the matrices whose eigenvectors the direct path leaves to its fallback.

Tolerance: a backward-stable reduction perturbs A by p(n) u ||A|| with p(n) of order n; n 2^-52
(2 n u) is taken for eigenvalues, residuals and orthonormality."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


def _sym(n, seed, scale=1.0):
    A = np.random.default_rng(seed).standard_normal((n, n))
    return scale * (A + A.T)


def _check(A, k, residual=True):
    n = len(A)
    w, Z = dfscf.eigh_lowest(A, k) if k < n else dfscf.eigh(A)
    w, Z = w.cpu().numpy(), Z.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    norm, tol = np.max(np.abs(ref)), n * 2.0 ** -52
    assert np.max(np.abs(w - ref[:k])) <= tol * norm
    assert np.max(np.abs(Z.T @ Z - np.eye(k))) <= tol
    if residual:
        assert np.max(np.abs(A @ Z - Z * w)) <= tol * norm


@pytest.mark.parametrize("n,k", [(32, 1), (33, 33), (47, 5), (127, 12), (128, 128), (129, 13), (146, 2), (255, 26),
                                 (257, 257), (512, 9), (513, 60), (1025, 30)])
def test_edges_of_tiles(n, k):
    _check(_sym(n, n + k), k)


@pytest.mark.parametrize("ctas", [2, 7, 33])
def test_rows_per_cta(ctas):
    dfscf.lib().df_tune_set(b"eig_ctas", ctas)
    try:
        _check(_sym(110, ctas), 17)
    finally:
        dfscf.lib().df_tune_set(b"eig_ctas", 0)


@pytest.mark.parametrize("scale", [1e-200, 1e-150, 1e150])
def test_far_from_one(scale):
    _check(_sym(70, 5, scale), 9)


@pytest.mark.parametrize("n", [50, 200])
@pytest.mark.parametrize("kind", ["graded", "equal blocks", "zero column", "diagonal", "identity", "nearly tridiagonal"])
def test_special_matrices(kind, n):
    rng = np.random.default_rng(n)
    X = _sym(n, n)
    if kind == "graded":
        Q, _ = np.linalg.qr(X)
        A = (Q * np.logspace(0, -12, n)) @ Q.T
    elif kind == "equal blocks":  # a pair of equal eigenvalues for each one of the block
        h = n // 2
        A = np.zeros((n, n))
        A[:h, :h] = A[h:2 * h, h:2 * h] = X[:h, :h]
    elif kind == "zero column":
        A = X
        A[0] = A[:, 0] = A[n // 2] = A[:, n // 2] = 0.0
    elif kind == "diagonal":
        A = np.diag(rng.standard_normal(n))
    elif kind == "identity":
        A = np.eye(n)
    else:
        A = np.diag(rng.standard_normal(n)) + np.diag(np.full(n - 1, 1e-3), 1) + np.diag(np.full(n - 1, 1e-3), -1)
    A = 0.5 * (A + A.T)
    for k in (n // 5, n):
        # equal eigenvalues go to inverse iteration, whose vectors of a cluster are less accurate
        _check(A, k, residual=kind not in ("equal blocks", "identity"))


def test_wait_that_runs_out_at_a_small_size():
    old = {name: dfscf.lib().df_tune_get(name) for name in (b"eig_barrier_extra", b"eig_barrier_polls")}
    try:
        dfscf.lib().df_tune_set(b"eig_barrier_polls", 4096)
        dfscf.lib().df_tune_set(b"eig_barrier_extra", 1)
        for call in (lambda A: dfscf.eigh_lowest(A, 4), dfscf.eigh):
            with pytest.raises(dfscf.DFError) as exc:
                call(_sym(60, 1))
            assert exc.value.code == dfscf.DF_ERR_TIMEOUT
    finally:
        for name, v in old.items():
            dfscf.lib().df_tune_set(name, v)
    torch.cuda.synchronize()
    _check(_sym(60, 1), 4)


def test_batch_with_one_slot():
    """Molecules one after another: the pass in which the last running one ends, before the next
    has started, is not a workspace too small."""
    import gen
    mols = [gen.make_molecule(n, gen.molecules.box_for(n), n) for n in (8, 5, 6)]
    batch = dfscf.scf_run_batch(mols, precision="fp64", slots=1)
    for m, r in zip(mols, batch.results):
        assert abs(r.energy - dfscf.scf_run(m, precision="fp64").energy) <= 1e-9

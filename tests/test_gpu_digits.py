"""The FP64 exchange on digit products (tensor cores) against extended precision.

K's sampled entries are compared with sums in numpy's long double (64 or more significand bits)
from the same B and C.  The bound: the two contractions each leave at most 2^-58 of (row max)
(column max) per 64-term chunk and are rounded to FP64, and K is the sum of the squares of
rounded X, so |dK_mn| <= 2^-52 sqrt(K_mm K_nn) with room for the split sums; a plain FP64 sum
may be off by more.  Sizes: one centre, edges of the 16/32-column groups, of the 128-row and
64-column tiles and of the 32/64-term stages, and more than one block of auxiliary rows."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
LD = np.longdouble


def sampled_k(B, C, rows):
    b = B.buf[:8 * B.naux * B.ld].view(torch.float64).view(B.naux, B.ld).cpu().numpy()
    n = np.arange(B.nao)
    R = np.stack([b[:, np.maximum(m, n) * (np.maximum(m, n) + 1) // 2 + np.minimum(m, n)] for m in rows], 1).astype(LD)
    X = np.stack([(R * C[:, i].astype(LD)).sum(2) for i in range(C.shape[1])], 2)
    return np.array([[(X[:, a] * X[:, c]).sum() for c in range(len(rows))] for a in range(len(rows))])


@pytest.fixture(scope="module")
def tensors():
    made = {}

    def get(n, nfun):
        if (n, nfun) not in made:
            mol = gen.molecule_from_geometry(gen.make_geometry(n, 2 * gen.molecules.box_for(n), 5),
                                             gen.even_tempered(0.1, 10.0, nfun))
            L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
            made[n, nfun] = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, "fp64")
        return made[n, nfun]

    return get


@pytest.mark.parametrize("n,nfun,nocc", [(1, 1, 1), (1, 5, 2), (7, 5, 16), (13, 5, 17), (16, 4, 33), (16, 4, 64),
                                         (26, 5, 65), (32, 4, 32), (43, 3, 9), (43, 5, 70)])
def test_exchange_against_extended_precision(tensors, n, nfun, nocc):
    B = tensors(n, nfun)
    rng = np.random.default_rng(nocc)
    C = rng.standard_normal((B.nao, nocc)) * np.exp(rng.uniform(-6, 3, (B.nao, 1)))
    _, K = dfscf.jk(B, None, C)
    rows = sorted({int(r) for r in np.linspace(0, B.nao - 1, 5)})
    ref = sampled_k(B, C, rows)
    scale = np.sqrt(np.outer(np.diag(ref), np.diag(ref)))
    err = np.abs(K.cpu().numpy()[np.ix_(rows, rows)].astype(LD) - ref) / scale
    assert float(err.max()) <= 2.0 ** -52 * 2
    assert torch.equal(K, K.T)


def test_exchange_blocks_and_splits_agree(tensors):
    """Other split counts and group widths change only the last rounding."""
    B = tensors(43, 5)
    C = np.random.default_rng(3).standard_normal((B.nao, 70))
    _, K = dfscf.jk(B, None, C)
    lib = dfscf.lib()
    try:
        for name, value in ((b"fp64_syrk_split", 1), (b"fp64_syrk_split", 13), (b"fp64_ht_cols", 16)):
            lib.df_tune_set(name, value)
            _, K2 = dfscf.jk(B, None, C)
            lib.df_tune_reset()
            assert float((K2 - K).abs().max()) <= 2.0 ** -50 * float(K.abs().max())
    finally:
        lib.df_tune_reset()


@pytest.mark.parametrize("value", [float("inf"), float("nan"), 5e-324])
def test_exchange_of_extreme_values(tensors, value):
    """Infinities and NaN come out where a plain sum has them; the smallest double does not
    disturb the other columns."""
    B = tensors(7, 5)
    C = torch.ones(B.nao, 3, dtype=torch.float64, device="cuda")
    C[4, 1] = value
    _, K = dfscf.jk(B, None, C)
    b = B.buf[:8 * B.naux * B.ld].view(torch.float64).view(B.naux, B.ld)
    i, j = np.tril_indices(B.nao)
    T = torch.zeros(B.naux, B.nao, B.nao, dtype=torch.float64, device="cuda")
    T[:, i, j] = b[:, :len(i)]
    T[:, j, i] = b[:, :len(i)]
    X = (T[:, :, :, None] * C[None, None]).sum(2).permute(1, 0, 2).reshape(B.nao, -1)
    ref = (X[:, None, :] * X[None]).sum(2)
    assert torch.equal(torch.isnan(K), torch.isnan(ref)) and torch.equal(torch.isinf(K), torch.isinf(ref))
    fine = torch.isfinite(ref)
    if fine.any():
        assert float((K - ref)[fine].abs().max()) <= 1e-13 * float(ref[fine].abs().max())

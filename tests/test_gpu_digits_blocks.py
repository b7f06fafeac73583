"""The FP64 exchange over several blocks of auxiliary rows, the last one shorter, with splits that
leave some without work, against extended precision.

Bound: the products of a block are exact sums rounded once, X is rounded once on either side, and
adding a block rounds the running sum, itself at most sqrt(K_mm K_nn): (4 + blocks) 2^-53 of that."""
import numpy as np
import pytest

import gen
from test_gpu_digits import LD, sampled_k

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


@pytest.mark.parametrize("pb,px,split", [(33, 100, 7), (17, 17, 1), (64, 129, 64), (1, 389, 3), (390, 390, 0)])
@pytest.mark.parametrize("nocc", [3, 65])
def test_uneven_blocks(pb, px, split, nocc):
    mol = gen.molecule_from_geometry(gen.make_geometry(26, 2 * gen.molecules.box_for(26), 5))
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    B = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, "fp64")
    assert B.naux == 390
    C = np.random.default_rng(nocc).standard_normal((B.nao, nocc))
    lib = dfscf.lib()
    try:
        for name, value in ((b"fp64_k_pb", pb), (b"fp64_k_px", px), (b"fp64_syrk_split", split)):
            assert lib.df_tune_set(name, value) == dfscf.DF_OK
        _, K = dfscf.jk(B, None, C)
    finally:
        lib.df_tune_reset()
    rows = sorted({int(r) for r in np.linspace(0, B.nao - 1, 5)})
    ref = sampled_k(B, C, rows)
    scale = np.sqrt(np.outer(np.diag(ref), np.diag(ref)))
    err = np.abs(K.cpu().numpy()[np.ix_(rows, rows)].astype(LD) - ref) / scale
    assert float(err.max()) <= (4 + -(-390 // max(px, pb))) * 2.0 ** -53

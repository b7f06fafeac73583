"""A workspace sized for more occupied columns serves fewer, also where its size is the smaller one.

Bound on K: its blocks are exact sums rounded once, X is rounded once on either side, adding a block
rounds the running sum: (4 + blocks) 2^-53 of sqrt(K_mm K_nn) on each of the two layouts; at most 3 blocks here."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


def workspace(nao, naux, nocc, nbytes):
    w = dfscf.JKWorkspace(nao, naux, 1, "fp64")
    w.key, w.buf = (nao, naux, nocc, 0), torch.full((nbytes + 512,), 0xA5, dtype=torch.uint8, device="cuda")[:nbytes]
    return w


@pytest.mark.parametrize("k,nocc", [(15, 64), (4, 33), (4, 57)])
def test_jk_with_fewer_columns(k, nocc):
    lib = dfscf.lib()
    mol = gen.molecule_from_geometry(gen.make_geometry(26, 2 * gen.molecules.box_for(26), 5),
                                     aux_exp=gen.even_tempered(0.1, 60.0, k))
    nao, naux = mol.nao, mol.naux
    sizes = {n: lib.df_jk_work_bytes(nao, naux, n, 0) for n in range(nocc, nao + 1)}
    least = min(sizes.values())
    assert least < sizes[nocc]
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    B = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, "fp64")
    C = np.random.default_rng(nocc).standard_normal((nao, nocc))
    D = 2 * C @ C.T
    J, K = (t.cpu().numpy() for t in dfscf.jk(B, D, C))
    scale = np.sqrt(np.outer(np.diag(K), np.diag(K)))
    w = workspace(nao, naux, nocc, least)
    J2, K2 = (t.cpu().numpy() for t in dfscf.jk(B, D, C, work=w))
    whole = torch.as_strided(w.buf, (512,), (1,), least)
    assert bool((whole == 0xA5).all())
    assert np.array_equal(J, J2)
    assert float((np.abs(K - K2) / scale).max()) <= 2 * (4 + 3) * 2.0 ** -53
    with pytest.raises(dfscf.DFError) as e:
        dfscf.jk(B, D, C, work=workspace(nao, naux, nocc, least - 1))
    assert e.value.code == dfscf.DF_ERR_NOMEM


def test_scf_with_fewer_columns(monkeypatch):
    """Two iterations: K differs by some 2^-53, which the density of the first passes on to the energy."""
    mol = gen.molecule_from_geometry(gen.make_geometry(40, gen.molecules.box_for(40), 3),
                                     aux_exp=gen.even_tempered(0.1, 2.0, 4))
    run = lambda: dfscf.scf_run(mol, precision="fp64", max_cycle=2, raise_on_noconv=False).energy
    size = dfscf.scf_work_bytes
    assert mol.nocc == 20 and size(mol.nao, mol.naux, 21) < size(mol.nao, mol.naux, 20)
    ref = run()
    monkeypatch.setattr(dfscf, "scf_work_bytes", lambda nao, naux, nocc, prec: size(nao, naux, 21, prec))
    assert abs(run() - ref) <= 1e-9 * abs(ref)

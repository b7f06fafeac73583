"""Workspaces of any alignment: with `work` 8 bytes past a 256-byte boundary, of exactly the size
the query gives, every entry point returns what it returns for an aligned one, and writes nothing
behind the workspace.  Same kernels on the same numbers: the results are equal bit for bit."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
GUARD = 512


class Workspaces:
    """Stand-in for the binding's allocator: tensors `shift` bytes past an aligned address."""

    def __init__(self, shift):
        self.shift, self.made = shift, []

    def __call__(self, nbytes):
        n = int(nbytes)
        buf = torch.full((n + self.shift + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
        assert buf.data_ptr() % 256 == 0
        self.made.append((buf, self.shift + n))
        return buf[self.shift:self.shift + n]

    def guards_whole(self):
        return all(bool((buf[end:] == 0xA5).all()) and bool((buf[:self.shift] == 0xA5).all()) for buf, end in self.made)


def results():
    from paper_2506_06661_gb300 import guess
    mol = gen.make_molecule(9, gen.molecules.box_for(9), 2)
    small = gen.molecule_from_geometry(gen.make_geometry(4, 5.0, 1), aux_exp=gen.even_tempered(0.1, 0.6, 2))
    C = np.random.default_rng(1).standard_normal((mol.nao, mol.nocc))
    Cs = C[:small.nao, :2].copy()
    A = np.random.default_rng(2).standard_normal((150, 150))
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    out = [L]
    for prec in ("fp64", "mixed"):
        B = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, prec)
        out += [B.buf[:8 * B.naux * B.ld], *dfscf.jk(B, 2 * C @ C.T, C, precision=prec)]
    out += [*dfscf.eigh(A + A.T), *dfscf.eigh_lowest(A + A.T, 11), *guess.lowdin_factors(mol)]
    out += list(dfscf.core_guess(mol)[:5])
    T = dfscf.lrdf_build(small.ao_xyz, small.ao_exp, small.aux_xyz, small.aux_exp, 0.4)
    out += [T.buf, *dfscf.lrdf_jk(T, small.ao_xyz, small.ao_exp, 0.4, 2 * Cs @ Cs.T, Cs)]
    k = np.tile(np.arange(15), mol.natm).astype(float)
    out += list(dfscf.fit_residual(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, k * mol.aux_exp)[:2])
    out.append(guess.predict_density(guess.GuessModel.create(seed=1), mol))
    for prec in ("fp64", "mixed"):
        out.append(dfscf.scf_run(mol, precision=prec).D)
    return out


def test_eight_byte_aligned_workspaces(monkeypatch):
    from paper_2506_06661_gb300 import guess
    ref = results()
    alloc = Workspaces(8)
    monkeypatch.setattr(dfscf, "_work", alloc)
    monkeypatch.setattr(guess, "_work", alloc)
    got = results()
    torch.cuda.synchronize()
    assert len(alloc.made) > 15 and alloc.guards_whole()
    for a, b in zip(ref, got):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


def test_batch_in_an_eight_byte_aligned_workspace():
    mols = [gen.make_molecule(n, gen.molecules.box_for(n), n) for n in (7, 4, 6)]
    need = dfscf.lib().scf_batch_work_bytes((dfscf.DFMolecule * 3)(*[dfscf.MoleculeOnDevice(m).c for m in mols]), 3, 0, 2)
    alloc = Workspaces(8)
    batch = dfscf.scf_run_batch(mols, precision="fp64", slots=2, work=alloc(need))
    ref = dfscf.scf_run_batch(mols, precision="fp64", slots=2)
    assert alloc.guards_whole()
    assert [r.energy for r in batch.results] == [r.energy for r in ref.results]

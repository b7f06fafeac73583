"""A wait of the tensor-core kernels that gives up is DF_ERR_TIMEOUT, whichever call it happens in.

Nothing waits here: the knob "tc_give_up" raises an error word from the host before the launches
(1: metric and whitening, 2: exchange), as a wait that gave up leaves it for the launches after
it, and the kernels skip their work.  The same calls give the same results as before afterwards."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


def code_of(call, hook):
    """The DFError code of a call made with the hook set."""
    assert dfscf.lib().df_tune_set(b"tc_give_up", hook) == dfscf.DF_OK
    try:
        with pytest.raises(dfscf.DFError) as exc:
            call()
    finally:
        dfscf.lib().df_tune_set(b"tc_give_up", 0)
    torch.cuda.synchronize()
    return exc.value.code


@pytest.fixture(scope="module")
def mol():
    return gen.make_molecule(9, gen.molecules.box_for(9), 2)


def test_set_up_calls(mol):
    args = (mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp)
    small = gen.molecule_from_geometry(gen.make_geometry(9, 8.0, 1), aux_exp=gen.even_tempered(0.1, 0.6, 4))
    lr = (small.ao_xyz, small.ao_exp, small.aux_xyz, small.aux_exp, 0.4)
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    T = dfscf.lrdf_build(*lr).buf
    assert code_of(lambda: dfscf.metric_chol(mol.aux_xyz, mol.aux_exp), 1) == dfscf.DF_ERR_TIMEOUT
    for prec in ("fp64", "mixed"):
        assert code_of(lambda: dfscf.build_B(*args, L, prec), 1) == dfscf.DF_ERR_TIMEOUT
    assert code_of(lambda: dfscf.lrdf_build(*lr), 1) == dfscf.DF_ERR_TIMEOUT
    assert code_of(lambda: dfscf.fit_residual(*args), 1) == dfscf.DF_ERR_TIMEOUT
    assert torch.equal(dfscf.metric_chol(mol.aux_xyz, mol.aux_exp), L) and torch.equal(dfscf.lrdf_build(*lr).buf, T)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_exchange(mol, prec):
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    B = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, prec)
    C = np.random.default_rng(0).standard_normal((mol.nao, 4))
    K = dfscf.jk(B, None, C, precision=prec)[1]
    out = torch.zeros_like(K)
    assert code_of(lambda: dfscf.jk(B, None, C, precision=prec, out_k=out), 2) == dfscf.DF_ERR_TIMEOUT
    assert bool(torch.isnan(out).all())
    assert torch.equal(dfscf.jk(B, None, C, precision=prec)[1], K)


@pytest.mark.parametrize("hook", [1, 2])  # set-up; first iteration
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_scf(mol, prec, hook):
    energy = dfscf.scf_run(mol, precision=prec).energy
    D0 = dfscf.core_guess(mol)[1] * 0.98  # not idempotent: the first exchange runs eagerly
    for dm0 in (None, D0):
        assert code_of(lambda: dfscf.scf_run(mol, dm0=dm0, precision=prec), hook) == dfscf.DF_ERR_TIMEOUT
    assert dfscf.scf_run(mol, precision=prec).energy == energy
    batch = []
    lib = dfscf.lib()
    lib.df_tune_set(b"tc_give_up", hook)
    try:
        batch = dfscf.scf_run_batch([mol, mol], precision=prec, slots=2, raise_on_noconv=False).results
    finally:
        lib.df_tune_set(b"tc_give_up", 0)
    assert not any(r.converged for r in batch)

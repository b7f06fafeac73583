"""Metric, Cholesky factor, three-centre integrals and whitening at the edges of their blocks (32 and
128 rows, 65536 columns), and the split weight gradients of the learned guess at batch edges.

Bounds.  Integrals: 28 FP64 roundings of 2^-53, a table error below 2^-53 and the oracle's own
give under 1e-14 relative to the largest.  L: backward error of a Cholesky factorisation,
|L L^T - M| <= (n + 1) 2^-53 |L| |L^T|.  B: backward error of the substitution, |L B - R| <=
(n + 1) 2^-53 |L| |B| entry by entry, the digit updates leaving no more than 2^-58 of row maximum
times column maximum per 64 terms, and underflow adding the smallest double per operation."""
import numpy as np
import pytest
import torch

import gen
import oracle

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
from paper_2506_06661_gb300 import guess  # noqa: E402


def rows_of(B):
    return B.buf[:8 * B.naux * B.ld].view(torch.float64).view(B.naux, B.ld)[:, :B.nao * (B.nao + 1) // 2].cpu().numpy()


def molecule(n, nfun, naux, box=1.0):
    """n centres with nfun orbital functions; naux auxiliary ones, spread over the centres."""
    xyz = gen.make_geometry(n, box * gen.molecules.box_for(n), 7)
    mol = gen.molecule_from_geometry(xyz, gen.even_tempered(0.1, 10.0, nfun))
    at = np.arange(naux) % n
    mol.aux_xyz = np.ascontiguousarray(xyz[at])
    mol.aux_exp = np.ascontiguousarray(0.1 * 3.0 ** (np.arange(naux) // n))
    return mol


@pytest.mark.parametrize("naux", [1, 31, 32, 33, 64, 65, 127, 128, 129, 161, 300])
def test_set_up_at_block_edges(naux):
    mol = molecule(60, 1, naux, box=2.0)
    L, M = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp, return_metric=True)
    Mo = oracle.int2c(mol.aux_xyz, mol.aux_exp)
    M, Ln = M.cpu().numpy(), L.cpu().numpy()
    assert np.max(np.abs(M - Mo)) <= 1e-14 * np.max(np.abs(Mo)) and np.array_equal(M, M.T)
    eps = (naux + 1) * 2.0 ** -53
    assert np.all(np.abs(Ln @ Ln.T - M) <= 2 * eps * (np.abs(Ln) @ np.abs(Ln).T))
    assert np.all(np.triu(Ln, 1) == 0.0)
    eye = torch.eye(naux, dtype=torch.float64, device="cuda")
    R = rows_of(dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, eye))
    Ro = oracle.int3c(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp)
    assert np.max(np.abs(R - Ro)) <= 1e-14 * np.max(np.abs(Ro))
    B = rows_of(dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L))
    floor = 2.0 ** -50 * np.max(np.abs(Ln), 1)[:, None] * np.max(np.abs(B), 0)[None] + 1000 * 5e-324
    assert np.all(np.abs(Ln @ B - R) <= 2 * eps * (np.abs(Ln) @ np.abs(B)) + floor)


def test_whitening_of_more_than_one_column_chunk():
    mol = molecule(74, 5, 150, box=2.0)  # 68635 pairs
    L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
    B = rows_of(dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L))
    R = rows_of(dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp,
                              torch.eye(150, dtype=torch.float64, device="cuda")))
    Ln = L.cpu().numpy()
    floor = 2.0 ** -50 * np.max(np.abs(Ln), 1)[:, None] * np.max(np.abs(B), 0)[None] + 1000 * 5e-324
    assert np.all(np.abs(Ln @ B - R) <= 302 * 2.0 ** -53 * (np.abs(Ln) @ np.abs(B)) + floor)


@pytest.mark.parametrize("t", [0.0, 1e-300, 1.0 / 64, 1.0 / 64 + 1e-12, 39.98, 39.9999999, 40.0, 41.0, 1e5])
def test_boys_table_edges(t):
    """(Q|mn) of coincident orbitals at distance R from Q is prefactor x F0(rho R^2)."""
    a, c = 0.7, 1.3
    rho = 2 * a * c / (2 * a + c)
    z = np.zeros((1, 3))
    q = np.array([[np.sqrt(t / rho), 0.0, 0.0]])
    B = dfscf.build_B(z, np.array([a]), q, np.array([c]), np.ones((1, 1)))
    ref = oracle.int3c(z, np.array([a]), q, np.array([c]))
    assert abs(rows_of(B)[0, 0] / ref.ravel()[0] - 1) <= 5e-15


@pytest.mark.parametrize("n", [1, 15, 64, 65, 1000])
def test_guess_gradient_at_batch_edges(n):
    """Split weight gradients against FP64 autograd; FP32 sums of n terms of like size."""
    g = torch.Generator().manual_seed(n)
    model = guess.GuessModel.create(seed=2)
    X, Y = torch.rand(n, 65, generator=g).cuda(), torch.randn(n, 15, generator=g).cuda()
    loss, grad = guess.loss_grad(model.params, X, Y)
    p, h, at = model.params.double().requires_grad_(True), X.double(), 0
    for k, (i, o) in enumerate(guess.LAYERS):
        h = h @ p[at:at + i * o].view(o, i).T + p[at + i * o:at + i * o + o]
        h = torch.nn.functional.silu(h) if k < 3 else h
        at += i * o + o
    ref = ((h - Y.double()) ** 2).mean()
    ref.backward()
    assert abs(loss - float(ref)) <= 1e-5 * float(ref)
    assert float((grad - p.grad).norm()) <= 1e-5 * float(p.grad.norm())

"""The work that users of the library have it do, as cases that can be timed and checked.

A case is one call sequence through the Python binding (paper_2506_06661_gb300), on synthetic
molecules of hydrogen-like centres with even-tempered s functions, 5 orbital and 15 auxiliary
ones on each centre.  Two densities are used: one centre per 10 bohr^3 (mixed SCFs) and one per
80 bohr^3 (single Fock builds, set-ups, FP64 SCFs), whose auxiliary metric is well enough
conditioned (about 1e11 instead of 1e16) for FP64 results to be determined to 1e-10.  The factor
of the metric itself is only determined to that with a sparser set, 8 auxiliary functions.
Mixed precision is timed as users run it, inside an SCF that ends in FP64: a single mixed
exchange matrix carries rounding noise of about 3e-8 that the last bits of its inputs move.
"""
import math

import numpy as np
import torch

import paper_2506_06661_gb300 as dfscf
from paper_2506_06661_gb300 import guess

LOOSE, DENSE = 80.0, 10.0  # bohr^3 per centre
F64 = torch.float64


def listed():
    return [
        # One Fock build (J and K) in FP64: a 20-centre molecule, where launches and latency count;
        # a ragged mid-size one; and a large one, where the exchange contractions are everything.
        {"name": "jk_fp64_20", "op": "jk", "centres": 20, "exchange": True},
        {"name": "jk_fp64_63", "op": "jk", "centres": 63, "exchange": True},
        {"name": "jk_fp64_200", "op": "jk", "centres": 200, "exchange": True},
        # The Coulomb matrix alone, as a response calculation or a pure functional asks for it.
        {"name": "j_fp64_120", "op": "jk", "centres": 120, "exchange": False},
        # Set-up of a molecule: three-centre integrals and whitening with a given factor of the
        # metric, and the metric with its Cholesky factor.
        {"name": "build_B_30", "op": "build_B", "centres": 30},
        {"name": "build_B_150", "op": "build_B", "centres": 150},
        {"name": "metric_chol_250", "op": "metric", "centres": 250},
        # The diagonalisation of each SCF iteration: the occupied orbitals and the next one.
        {"name": "eigh_lowest_900", "op": "eigh", "n": 900, "k": 91},
        # A whole FP64 SCF of a small molecule, a mixed-precision one of a mid-size molecule, and a
        # batch of uneven molecules in mixed precision.
        {"name": "scf_fp64_20", "op": "scf", "precision": "fp64", "centres": 20},
        {"name": "scf_mixed_60", "op": "scf", "precision": "mixed", "centres": 60},
        {"name": "scf_batch_mixed_8", "op": "batch", "molecules": 8, "smallest": 10, "largest": 40},
        # One training step (forward, backward, Adam) of the learned initial guess.
        {"name": "guess_train_4096", "op": "train", "pairs": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["jk", "jk", "jk", "build_B", "build_B", "metric", "eigh", "scf", "scf", "batch", "train"])
    if op == "jk":
        return {"op": op, "centres": _log_int(rng, 10, 190), "exchange": rng.random() < 0.8}
    if op == "build_B":
        return {"op": op, "centres": _log_int(rng, 10, 140)}
    if op == "metric":
        return {"op": op, "centres": _log_int(rng, 20, 240)}
    if op == "eigh":
        n = _log_int(rng, 50, 900)
        return {"op": op, "n": n, "k": n // 10 + 1}
    if op == "scf":
        precision = rng.choice(["fp64", "mixed"])
        return {"op": op, "precision": precision, "centres": rng.randint(8, 24) if precision == "fp64" else _log_int(rng, 12, 55)}
    if op == "batch":
        return {"op": op, "molecules": rng.randint(3, 8), "smallest": rng.randint(8, 12), "largest": rng.randint(18, 38)}
    return {"op": op, "pairs": _log_int(rng, 300, 8192)}


# ---- molecules ---------------------------------------------------------------------------
class Molecule:
    """Arrays of one molecule, as MoleculeOnDevice takes them."""

    def __init__(self, n, volume, seed, aux=0.05 * 1000.0 ** (np.arange(15) / 14)):
        rng = np.random.default_rng(seed)
        box, pts = (volume * n) ** (1.0 / 3.0), np.empty((0, 3))
        while len(pts) < n:  # uniform in a cube, no two centres within 1.4 bohr
            p = rng.uniform(0.0, box, 3)
            if not len(pts) or np.min(np.sum((pts - p) ** 2, 1)) >= 1.96:
                pts = np.vstack([pts, p])
        orb = 0.1 * 100.0 ** (np.arange(5) / 4)
        self.xyz, self.charges, self.natm = pts, np.ones(n), n
        self.ao_xyz, self.ao_exp, self.nao = np.repeat(pts, 5, 0), np.tile(orb, n), 5 * n
        self.aux_xyz, self.aux_exp, self.naux = np.repeat(pts, len(aux), 0), np.tile(aux, n), len(aux) * n
        self.nelec = n - n % 2


def _cuda(x):
    return torch.as_tensor(x, dtype=F64).cuda()


# ---- closed forms of the s integrals in plain torch ----------------------------------------
def _boys(t):
    s = torch.sqrt(t.clamp_min(1e-30))
    small = 1 - t * (1 / 3 - t * (1 / 10 - t * (1 / 42 - t * (1 / 216 - t / 1320))))
    return torch.where(t < 1e-3, small, 0.5 * math.sqrt(math.pi) * torch.erf(s) / s)


def _norm(a):
    return (2 * a / math.pi) ** 0.75


def _pairs(xyz, ex):
    """(exponent sum, centre, N_a N_b exp(-mu R^2)) of the packed pairs m >= n."""
    m, n = np.tril_indices(len(ex))
    m, n = torch.as_tensor(m, device=ex.device), torch.as_tensor(n, device=ex.device)
    p = ex[m] + ex[n]
    r2 = ((xyz[m] - xyz[n]) ** 2).sum(1)
    return p, (ex[m, None] * xyz[m] + ex[n, None] * xyz[n]) / p[:, None], \
        _norm(ex[m]) * _norm(ex[n]) * torch.exp(-ex[m] * ex[n] / p * r2)


def _full(packed, n):
    A = torch.zeros(n, n, dtype=F64, device=packed.device)
    i, j = np.tril_indices(n)
    A[i, j] = packed
    A[j, i] = packed
    return A


def _overlap(xyz, ex):
    p, _, k = _pairs(xyz, ex)
    return _full(k * (math.pi / p) ** 1.5, len(ex))


def _core(mol):
    """S and h = T + V."""
    xyz, ex, nuc = _cuda(mol.ao_xyz), _cuda(mol.ao_exp), _cuda(mol.xyz)
    p, c, k = _pairs(xyz, ex)
    m, n = np.tril_indices(mol.nao)
    mu = ex[m] * ex[n] / p
    s = k * (math.pi / p) ** 1.5
    t = mu * (3 - 2 * mu * ((xyz[m] - xyz[n]) ** 2).sum(1)) * s
    v = torch.zeros_like(s)
    for a in nuc:
        v -= 2 * math.pi / p * k * _boys(p * ((c - a) ** 2).sum(1))
    return _full(s, mol.nao), _full(t + v, mol.nao)


def _metric(mol):
    xyz, ex = _cuda(mol.aux_xyz), _cuda(mol.aux_exp)
    s = ex[:, None] + ex[None]
    r2 = ((xyz[:, None] - xyz[None]) ** 2).sum(2)
    pre = _norm(ex)[:, None] * _norm(ex)[None] * 2 * math.pi ** 2.5 / (ex[:, None] * ex[None] * torch.sqrt(s))
    return pre * _boys(ex[:, None] * ex[None] / s * r2)


def _three_centre(mol, lo, hi):
    """(Q|mn) for the packed pairs lo..hi."""
    p, c, k = (x[lo:hi] for x in _pairs(_cuda(mol.ao_xyz), _cuda(mol.ao_exp)))
    q, x = _cuda(mol.aux_exp)[:, None], _cuda(mol.aux_xyz)
    r2 = ((x[:, None, 0] - c[None, :, 0]) ** 2 + (x[:, None, 1] - c[None, :, 1]) ** 2 + (x[:, None, 2] - c[None, :, 2]) ** 2)
    return k[None] * _norm(q) * 2 * math.pi ** 2.5 / (p[None] * q * torch.sqrt(p[None] + q)) * _boys(p[None] * q / (p[None] + q) * r2)


def _whitened(mol, L):
    np_, step = mol.nao * (mol.nao + 1) // 2, 65536
    return torch.cat([torch.linalg.solve_triangular(L, _three_centre(mol, i, min(np_, i + step)), upper=False)
                      for i in range(0, np_, step)], 1)


def _orbitals(mol, seed):
    """Random orthonormal orbitals (C^T S C = 1) and their closed-shell density."""
    nocc = max(1, mol.nelec // 2)
    w, U = torch.linalg.eigh(_overlap(_cuda(mol.ao_xyz), _cuda(mol.ao_exp)))
    g = torch.Generator().manual_seed(seed)
    Q, _ = torch.linalg.qr(torch.randn(mol.nao, nocc, generator=g, dtype=F64).cuda())
    C = (U @ ((U.T @ Q) / torch.sqrt(w)[:, None])).contiguous()
    return C, (2 * C @ C.T).contiguous()


def _jk(B, nao, C, D):
    """J and K of packed rows B, auxiliary rows in slices."""
    i, j = (torch.as_tensor(x, device=B.device) for x in np.tril_indices(nao))
    w = torch.where(i == j, 1.0, 2.0).to(F64)
    J = _full((B @ (w * D[i, j])) @ B, nao)
    K = torch.zeros(nao, nao, dtype=F64, device=B.device)
    for p in range(0, B.shape[0], 64):
        T = torch.zeros(min(64, B.shape[0] - p), nao, nao, dtype=F64, device=B.device)
        T[:, i, j] = B[p:p + 64]
        T[:, j, i] = B[p:p + 64]
        X = (T @ C).permute(1, 0, 2).reshape(nao, -1)
        K += X @ X.T
    return J, K


def _rhf_energy(mol):
    """Closed-shell density-fitted Hartree-Fock energy from the core guess, with DIIS."""
    S, h = _core(mol)
    B = _whitened(mol, torch.linalg.cholesky(_metric(mol)))
    w, U = torch.linalg.eigh(S)
    X = U[:, w > 1e-8] / torch.sqrt(w[w > 1e-8])
    r = torch.sqrt(((_cuda(mol.xyz)[:, None] - _cuda(mol.xyz)[None]) ** 2).sum(2))
    e_nuc = float((1 / r[np.tril_indices(mol.natm, -1)]).sum())
    F, Fs, Es, old = h, [], [], 0.0
    for _ in range(200):
        C = (X @ torch.linalg.eigh(X.T @ F @ X)[1][:, :mol.nelec // 2]).contiguous()
        D = 2 * C @ C.T
        J, K = _jk(B, mol.nao, C, D)
        F = h + J - K
        E = 0.5 * float((D * (h + F)).sum()) + e_nuc
        err = X.T @ (F @ D @ S - S @ D @ F) @ X
        if abs(E - old) < 1e-10 and float(err.abs().max()) < 1e-6:
            break
        old, Fs, Es = E, (Fs + [F])[-8:], (Es + [err])[-8:]
        n = len(Fs)
        A = -torch.ones(n + 1, n + 1, dtype=F64, device="cuda")
        A[:n, :n] = torch.stack([torch.stack([(a * b).sum() for b in Es]) for a in Es])
        A[n, n] = 0
        b = torch.zeros(n + 1, dtype=F64, device="cuda")
        b[n] = -1
        F = sum(c * f for c, f in zip(torch.linalg.lstsq(A.cpu(), b.cpu()[:, None], driver="gelsd").solution[:n, 0].tolist(), Fs))
    return E


# ---- the cases -----------------------------------------------------------------------------
def _batch(case, seed):
    """Uneven molecules: sizes evenly spread over the range, so that every seed costs alike."""
    sizes = np.linspace(case["smallest"], case["largest"], case["molecules"]).round().astype(int)
    return [Molecule(int(n), DENSE, (seed, i)) for i, n in enumerate(sizes)]


def _symmetric(case, seed):
    """A matrix with the spectrum of a Fock matrix: occupied levels below a gap, virtual ones above."""
    n, k = case["n"], case["k"]
    g = torch.Generator().manual_seed(seed)
    w = torch.cat([torch.sort(-1.5 + 1.2 * torch.rand(k - 1, generator=g, dtype=F64))[0],
                   torch.sort(0.1 + 30 * torch.rand(n - k + 1, generator=g, dtype=F64) ** 2)[0]])
    Q, _ = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=F64).cuda())
    A = (Q * w.cuda()) @ Q.T
    return (0.5 * (A + A.T)).contiguous()


LAYERS = [(65, 256), (256, 256), (256, 256), (256, 15)]


def _training_set(case, seed):
    """(parameters, features, targets): a network's start and a mini-batch of pairs of random
    geometries (radial functions of the distance and of both surroundings, diagonal flag)."""
    g = torch.Generator().manual_seed(seed)
    params = torch.cat([torch.cat([(2 * torch.rand(o * i, generator=g) - 1) * math.sqrt(3 / i), torch.zeros(o)])
                        for i, o in LAYERS]).cuda()
    rows, n, centres = [], 0, torch.arange(32) * 12.0 / 31
    while n < case["pairs"]:
        xyz = torch.as_tensor(Molecule(30, DENSE, (seed, n)).xyz, dtype=torch.float32)
        r = torch.cdist(xyz, xyz)
        f = torch.exp(-((r[:, :, None] - centres) * 31 / 12) ** 2)
        f[torch.arange(30), torch.arange(30)] = 0
        env = f.sum(1) / 8
        a, b = np.tril_indices(30)
        rows.append(torch.cat([f[a, b], env[a] + env[b], torch.as_tensor(a == b, dtype=torch.float32)[:, None]], 1))
        n += len(a)
    X = torch.cat(rows)[torch.randperm(n, generator=g)[:case["pairs"]]].cuda().contiguous()
    return params, X, torch.tanh(0.2 * X @ torch.randn(65, 15, generator=g).cuda()).contiguous()


def _gradient(params, X, Y):
    """Loss and its gradient in 64 bits."""
    p, h, at = params.double().requires_grad_(True), X.double(), 0
    for k, (i, o) in enumerate(LAYERS):
        h = h @ p[at:at + i * o].view(o, i).T + p[at + i * o:at + i * o + o]
        h = torch.nn.functional.silu(h) if k < 3 else h
        at += i * o + o
    loss = ((h - Y.double()) ** 2).mean()
    loss.backward()
    return float(loss), p.grad


def _metric_molecule(case, seed):
    return Molecule(case["centres"], LOOSE, seed, 0.1 * 200.0 ** (np.arange(8) / 7))


def prepare(case, seed):
    op = case["op"]
    if op == "jk":
        mol = Molecule(case["centres"], LOOSE, seed)
        L = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp)
        B = dfscf.build_B(mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp, L, "fp64")
        C, D = _orbitals(mol, seed)
        work = dfscf.JKWorkspace(mol.nao, mol.naux, C.shape[1] if case["exchange"] else 0, "fp64")
        return op, B, C if case["exchange"] else None, D, work
    if op == "build_B":
        mol = Molecule(case["centres"], LOOSE, seed)
        arrays = [_cuda(x) for x in (mol.ao_xyz, mol.ao_exp, mol.aux_xyz, mol.aux_exp)]
        return (op, *arrays, torch.linalg.cholesky(_metric(mol)).contiguous())
    if op == "metric":
        mol = _metric_molecule(case, seed)
        return op, _cuda(mol.aux_xyz), _cuda(mol.aux_exp)
    if op == "eigh":
        return op, _symmetric(case, seed), case["k"]
    if op == "scf":
        mol = Molecule(case["centres"], LOOSE if case["precision"] == "fp64" else DENSE, seed)
        return op, dfscf.MoleculeOnDevice(mol), case["precision"]
    if op == "batch":
        return op, [dfscf.MoleculeOnDevice(m) for m in _batch(case, seed)]
    params, X, Y = _training_set(case, seed)
    return op, guess.GuessModel(params, torch.zeros_like(params), torch.zeros_like(params), 0), X, Y


def run(state):
    op = state[0]
    if op == "jk":
        _, B, C, D, work = state
        J, K = dfscf.jk(B, D, C, work=work)
        return {"J": J, "K": K} if K is not None else {"J": J}
    if op == "build_B":
        _, ao_xyz, ao_exp, aux_xyz, aux_exp, L = state
        B = dfscf.build_B(ao_xyz, ao_exp, aux_xyz, aux_exp, L, "fp64")
        return {"B": B.buf.view(F64)[:B.naux * B.ld].view(B.naux, B.ld)[:, :B.nao * (B.nao + 1) // 2]}
    if op == "metric":
        return {"L": dfscf.metric_chol(state[1], state[2])}
    if op == "eigh":
        w, Z = dfscf.eigh_lowest(state[1], state[2])
        return {"w": w, "P": Z[:, :-1] @ Z[:, :-1].T}
    if op == "scf":
        r = dfscf.scf_run(state[1], precision=state[2], raise_on_noconv=False)
        # a mixed run's density is that of its convergence threshold (1e-5), its energy to second order
        energy = np.array(r.energy)
        return {"energy": energy, "D": r.D, "mo_energy": r.mo_energy} if state[2] == "fp64" else {"energy": energy}
    if op == "batch":
        r = dfscf.scf_run_batch(state[1], precision="mixed", raise_on_noconv=False)
        return {"energy": np.array([x.energy for x in r.results])}
    _, model, X, Y = state
    loss, grad = guess.loss_grad(model.params, X, Y)
    guess.train(model, X, Y, torch.ones(len(X), device="cuda"), epochs=1, batch=len(X))
    return {"grad": grad, "loss": loss, "params": model.params}


def exact(case, seed):
    op = case["op"]
    if op == "jk":
        mol = Molecule(case["centres"], LOOSE, seed)
        C, D = _orbitals(mol, seed)
        J, K = _jk(_whitened(mol, torch.linalg.cholesky(_metric(mol))), mol.nao, C, D)
        return {"J": J, "K": K} if case["exchange"] else {"J": J}
    if op == "build_B":
        mol = Molecule(case["centres"], LOOSE, seed)
        return {"B": _whitened(mol, torch.linalg.cholesky(_metric(mol)))}
    if op == "metric":
        return {"L": torch.linalg.cholesky(_metric(_metric_molecule(case, seed)))}
    if op == "eigh":
        w, U = torch.linalg.eigh(_symmetric(case, seed))
        k = case["k"]
        return {"w": w[:k], "P": U[:, :k - 1] @ U[:, :k - 1].T}
    if op == "scf":
        if case["precision"] == "mixed":
            return {"energy": np.array(_rhf_energy(Molecule(case["centres"], DENSE, seed)))}
        return {"energy": np.array(_rhf_energy(Molecule(case["centres"], LOOSE, seed))), "D": None, "mo_energy": None}
    if op == "batch":
        return {"energy": np.array([_rhf_energy(m) for m in _batch(case, seed)])}
    params, X, Y = _training_set(case, seed)
    loss, g = _gradient(params, X, Y)
    return {"grad": g, "loss": loss, "params": params.double() - 1e-3 * g / (g.abs() + 1e-8)}


def work(case):
    op = case["op"]
    if op in ("jk", "build_B", "scf"):
        n = case["centres"]
    if op == "jk":
        return _jk_work(n, case["exchange"])
    if op == "build_B":
        npair, naux = 5 * n * (5 * n + 1) // 2, 15 * n
        return {"bytes": 8.0 * naux * (npair + naux / 2), "flops": float(naux) ** 2 * npair}
    if op == "metric":
        return {"bytes": 8.0 * (8 * case["centres"]) ** 2, "flops": (8.0 * case["centres"]) ** 3 / 3}
    if op == "eigh":
        n, k = case["n"], case["k"]
        return {"bytes": 8.0 * (n * n + n * k), "flops": 4.0 * n ** 3 / 3 + 2.0 * n * n * k}
    if op == "scf":
        return _scf_work(n)
    if op == "batch":
        sizes = np.linspace(case["smallest"], case["largest"], case["molecules"])
        each = [_scf_work(float(n)) for n in sizes]
        return {"bytes": sum(w["bytes"] for w in each), "flops": sum(w["flops"] for w in each)}
    layers = 65 * 256 + 2 * 256 * 256 + 256 * 15
    return {"bytes": 4.0 * (case["pairs"] * 80 * 2 + 8 * layers), "flops": 12.0 * case["pairs"] * layers}


def _jk_work(n, exchange=True):
    nao, naux, nocc = 5 * n, 15 * n, max(1, n // 2)
    npair = nao * (nao + 1) / 2
    j = {"bytes": 8.0 * (naux * npair + 2 * nao * nao), "flops": 4.0 * naux * npair}
    if not exchange:
        return j
    return {"bytes": j["bytes"] + 8.0 * (nao * nao + nao * nocc),
            "flops": j["flops"] + 2.0 * naux * nao * nao * nocc + 2.0 * naux * nocc * npair}


def _scf_work(n):
    """Whitening and, as about what such a molecule takes, 20 Fock builds and diagonalisations."""
    one, nao = _jk_work(int(n)), 5.0 * n
    return {"bytes": 20 * one["bytes"], "flops": 20 * (one["flops"] + 2 * nao ** 3) + (15.0 * n) ** 2 * nao * nao / 2}

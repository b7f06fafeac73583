"""The Coulomb metric is no further from the exact integrals than the closed form
N_c N_d 2 pi^{5/2} / (c d sqrt(c + d)) F0(cd/(c+d) R^2) evaluated in FP64 with erf is: both are
compared with the same expression in numpy's long double (root mean square of the relative errors)."""
import math

import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def boys_exact(t):
    """F0 by its series of positive terms below 46, where erf(sqrt t) is not 1 to long double."""
    out = np.sqrt(PI / np.where(t > 46, t, 1)) / 2
    x = t[t <= 46]
    term = np.ones_like(x)
    total = term.copy()
    for i in range(1, 260):
        term = term * (2 * x) / (2 * i + 1)
        total += term
    out[t <= 46] = np.exp(-x) * total
    return out


def boys_fp64(t):
    def f(x):
        if x < 1e-3:
            return 1 - x * (1 / 3 - x * (1 / 10 - x * (1 / 42 - x * (1 / 216 - x / 1320))))
        return 0.5 * math.sqrt(math.pi) * math.erf(math.sqrt(x)) / math.sqrt(x)
    return np.vectorize(f)(t)


def metric(xyz, ex, pi, boys):
    norm = (2 * ex / pi) ** (ex.dtype.type(3) / 4)
    s, cd = ex[:, None] + ex, ex[:, None] * ex
    r2 = ((xyz[:, None] - xyz) ** 2).sum(2)
    return norm[:, None] * norm * 2 * pi ** 2 * np.sqrt(pi) / (cd * np.sqrt(s)) * boys(cd / s * r2)


@pytest.mark.parametrize("centres,box,seed", [(10, 1.0, 1), (10, 2.0, 2), (12, 2.0, 3)])
def test_metric(centres, box, seed):
    mol = gen.make_molecule(centres, box * gen.molecules.box_for(centres), seed)
    ref = metric(mol.aux_xyz.astype(LD), mol.aux_exp.astype(LD), PI, boys_exact)
    plain = metric(mol.aux_xyz, mol.aux_exp, np.float64(math.pi), boys_fp64)
    _, M = dfscf.metric_chol(mol.aux_xyz, mol.aux_exp, return_metric=True)

    def rms(x):
        return float(np.sqrt((((x.astype(LD) - ref) / ref) ** 2).mean()))

    assert rms(M.cpu().numpy()) <= rms(plain)

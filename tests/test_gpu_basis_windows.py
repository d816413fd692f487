"""Basis integrals with few k nodes over five decades of k, against the oracle.

1/k^2 falls by up to 1e10 between neighbouring nodes there while j_l j_l rises,
so a digit's scale must not be shared by nodes far apart.  Both sides sum at most
1025 products with a rounding each, of Bessel functions from recurrences of some
fifty steps and T_n to order 3: 1e-14 of the sum of the products' magnitudes, j_l
at its envelope past x = l, holds each (random roundings: sqrt(1025) 2^-54 = 2e-15
and a few 1e-15 for the factors).
"""
import numpy as np
import pytest
from scipy.special import spherical_jn

import oracle as orc
from paper_2410_03632_gb300 import blast as bl
from paper_2410_03632_gb300 import synth

pytestmark = pytest.mark.gpu


def _have_gpu():
    try:
        import torch
        return torch.cuda.is_available()
    except Exception:
        return False


if not _have_gpu():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _envelope(l, x):
    return np.where(x > l, 1.0 / x, np.abs(spherical_jn(l, x)))


@pytest.mark.parametrize("chi_lo,chi_hi", [(1.0, 9.0), (20.0, 60.0)])
@pytest.mark.parametrize("nk", [5, 17, 65, 257, 1025])
def test_few_nodes(nk, chi_lo, chi_hi):
    ells = np.array([2, 5, 10], np.int32)
    spec = synth.PlanSpec(ells, 4, chi_lo, chi_hi, 6, 0.5, 1.5, 4, 1e-4, 10.0, 1, nk, 1, 1)
    g = orc.Grid(ells, 4, chi_lo, chi_hi, 6, 0.5, 1.5, 4, 1e-4, 10.0, nk, 1)
    plan = bl.Plan(spec)
    plan.precompute(bl.BLAST_BASIS_FP64)
    T = plan.basis()
    plan.close()
    ref = g.basis().reshape(T.shape)
    k, _, w = orc.cc_grid(nk, 1e-4, 10.0)
    c1, c2 = np.repeat(g.chi, 6), (g.chi[:, None] * g.R).ravel()
    for t, p in enumerate((2, 0, -2)):
        for e, l in enumerate(ells):
            size = (w * k ** float(p)) @ (_envelope(l, k[:, None] * c1) * _envelope(l, k[:, None] * c2))
            err = np.max(np.abs(T[t, e] - ref[t, e]) / size)
            assert err < 1e-14, (t, l, err)

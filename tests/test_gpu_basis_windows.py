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


def test_many_nodes_take_bounded_memory():
    """The digits are made part by part (four here): the build holds less than the FP64 A[k node][3 N]
    alone would take (403 MB).  The k sum has 131,073 terms, sqrt(131073) 2^-54 = 2e-14 for a chain of
    random roundings: 1e-13 of the sum of magnitudes."""
    import threading
    import time

    import torch

    N, nk = 128, 2 ** 17 + 1
    ells = np.array([2, 40], np.int32)
    spec = synth.PlanSpec(ells, 4, 300.0, 4100.0, 2, 0.5, 1.5, N, 1e-4, 10.0, 1, nk, 1, 1)
    plan = bl.Plan(spec)
    plan.precompute(bl.BLAST_BASIS_FP64)    # tables and code are in place
    T = plan.basis()
    free0, done, least = torch.cuda.mem_get_info()[0], threading.Event(), []
    worker = threading.Thread(target=lambda: (plan.precompute(bl.BLAST_BASIS_FP64), done.set()))
    worker.start()
    while not done.is_set():
        least.append(torch.cuda.mem_get_info()[0])
        time.sleep(1e-3)
    worker.join()
    np.testing.assert_array_equal(plan.basis(), T)
    plan.close()
    took = free0 - min(least)
    assert 0 < took < 24 * N * nk, took
    g = orc.Grid(ells, 4, 300.0, 4100.0, 2, 0.5, 1.5, N, 1e-4, 10.0, nk, 1)
    ref = g.basis().reshape(T.shape)
    k, _, w = orc.cc_grid(nk, 1e-4, 10.0)
    c1, c2 = np.repeat(g.chi, 2), (g.chi[:, None] * g.R).ravel()
    for t, p in enumerate((2, 0, -2)):
        for e, l in enumerate(ells):
            size = (w * k ** float(p)) @ (_envelope(l, k[:, None] * c1) * _envelope(l, k[:, None] * c2))
            assert np.max(np.abs(T[t, e, :4] - ref[t, e, :4]) / size) < 1e-13, (t, l)


def test_recurrences_out_of_range_are_not_numbers():
    """At distances of 1e-24 the downward recurrence of l = 40's group overflows: those integrals are NaN,
    the others (chi^4 k^5 and less: 1e-88) stay what they are, and no made-up number stands between."""
    spec = synth.PlanSpec(np.array([2, 3, 40], np.int32), 4, 1e-24, 4e-24, 4, 0.5, 1.5, 3, 1e-2, 10.0, 1, 65, 1, 1)
    plan = bl.Plan(spec)
    plan.precompute(bl.BLAST_BASIS_FP64)
    T = plan.basis()
    plan.close()
    bad = np.isnan(T)
    assert bad.any() and not bad.all()
    assert np.all(np.abs(T[~bad]) < 1e-60)

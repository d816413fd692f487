"""FP64 contraction of tables that rise with the order while the coefficients fall.

The digits are relative to max |a| max |T| of a column, a multiply-add chain to
its partial sums, so this is where the two paths differ most.  A second plan
whose table has an infinity in one more ell runs the multiply-add kernel; the
common spectra differ by the digits' error (about 2^-59 max |a| max |T|, digits of
random sign; 2^-56 taken) and the roundings both sides make, N + n_R + n_chi of
them at 2^-53 of the sum of magnitudes.  2^-56 is an eighth of what the fit rounds
every coefficient by, so no spectrum loses accuracy to the digits.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("N", [64, 96])
@pytest.mark.parametrize("rise", [1.0, 1e3, 1e6, 1e9])
def test_digits_against_multiply_adds(N, rise):
    X, Rn, ng, ns = 5, 64, 2, 2
    ells = np.array([2, 40, 300, 500], np.int32)
    rng = np.random.default_rng(N)
    T = rng.standard_normal((3, 4, N, X * Rn)) * (rise ** (np.arange(N) / (N - 1)))[:, None]
    T[0, 3, 0, 0] = np.inf
    k = np.geomspace(1e-4, 1.0, 256)
    P = 1e4 * np.exp(-2.0 * (2.0 * np.log(k / 1e-4) / np.log(1e4) - 1.0) ** 2)   # a_n falls by 1e9 and more
    rq = synth.Request(ng, ns, rng.random((4, X)), rng.random((4, X * Rn)), rng.random(X), rng.random(X * Rn), k, P)
    out = []
    for L in (3, 4):
        plan = bl.Plan(synth.PlanSpec(ells[:L], X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 1, 257, ng, ns))
        plan.set_basis(T[:, :L], bl.BLAST_BASIS_FP64)
        out.append(plan.cl(rq, bl.BLAST_FP64)[:, :3])
        plan.close()
    g = orc.Grid(ells[:3], X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 257, 1)
    a = np.abs(g.fit(k, P))
    args = (ng, ns, rq.kern_chi, rq.kern_Rchi, rq.growth_chi, rq.growth_Rchi)
    A = np.abs(T[:, :3])
    top = np.zeros_like(A)
    top[:, :, 0] = A.max(axis=2)
    size, most = g.cl(A, a, *args), g.cl(top, np.r_[a.max(), np.zeros(N - 1)], *args)
    assert np.all(np.abs(out[0] - out[1]) <= 2.0 ** -56 * most + (N + Rn + X) * 2.0 ** -53 * size)
    if rise == 1e6:  # and the bound is the digits', not the chain's
        assert np.max(np.abs(out[0] - out[1]) / size) > 1e-14

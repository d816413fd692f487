"""Real multipoles at the top of the accepted range: eight recurrences of 1e5
steps a chain keep the build's warps waiting for seconds, which is no failure.
j_l comes from up to 1e5 + 484 steps of three roundings each (2^-53 a rounding:
3.4e-11 a factor at most, 7e-11 a product) at x known to 2^-53 (1e5 2^-53 = 1e-11
of the phase): 1e-9 of the sum of the products' envelopes."""
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


def test_build_at_the_largest_real_multipoles():
    ells = 99990.5 + np.arange(8)
    grid = (4, 0.8e5, 1.25e5, 8, 0.9, 1.1, 2, 0.9, 1.1)
    plan = bl.Plan(synth.PlanSpec(ells, *grid, 1, 65, 1, 1))
    plan.precompute(bl.BLAST_BASIS_FP64)
    T = plan.basis()
    plan.close()
    g = orc.Grid(ells, *grid, 65, 1)
    ref = g.basis().reshape(T.shape)
    k, _, w = orc.cc_grid(65, 0.9, 1.1)
    for t, p in enumerate((2, 0, -2)):
        size = w @ k ** (p - 2.0) / (np.repeat(g.chi, 8) * (g.chi[:, None] * g.R).ravel())
        assert np.max(np.abs(T[t] - ref[t]) / size) < 1e-9
        assert np.max(np.abs(T[t]) / size) > 1e-3      # the integrals are not empty

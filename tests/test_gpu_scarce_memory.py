"""Calls that still succeed when little device memory is left beside the plan."""
import numpy as np
import pytest

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


class _Only:
    """All but `left` bytes of the device's free memory taken."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        import torch
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.block = torch.empty(free - self.left, dtype=torch.uint8, device="cuda")

    def __exit__(self, *_):
        import torch
        del self.block
        torch.cuda.empty_cache()


def test_basis_build_takes_smaller_parts():
    """A part takes 270 MB at order 128; with 150 MB the build takes smaller ones, to the same bits."""
    spec = synth.PlanSpec(np.array([2, 40], np.int32), 4, 300.0, 4100.0, 2, 0.5, 1.5, 128, 1e-4, 10.0, 1, 2 ** 17 + 1,
                          1, 1)
    plan = bl.Plan(spec)
    plan.precompute(bl.BLAST_BASIS_FP64)
    T = plan.basis()
    with _Only(150 << 20):
        plan.precompute(bl.BLAST_BASIS_FP64)
    np.testing.assert_array_equal(plan.basis(), T)
    plan.close()


def test_table_without_room_for_its_exponents():
    """A table that fits is taken and evaluated by multiply-adds; every term is positive and each side rounds
    n_cheb + n_R + n_chi of them at 2^-53, after fits good to a few units."""
    X, Rn, N = 13100, 512, 2
    Q = X * Rn
    spec = synth.PlanSpec(np.array([2], np.int32), X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 1, 17, 1, 1)
    rng = np.random.default_rng(0)
    T = rng.random((3, 1, N, Q))
    T[:, :, 1] *= 1e-3                       # a_0 > 0 leads
    k, P = synth.pk_table(-2.0, 0.05, 0.0, 0.8)
    rq = synth.Request(1, 1, rng.random((2, X)), rng.random((2, Q)), rng.random(X), rng.random(Q), k, P)
    plan = bl.Plan(spec)
    plan.set_basis(T, bl.BLAST_BASIS_FP64)
    ref = plan.cl(rq, bl.BLAST_FP64)
    plan.close()
    plan = bl.Plan(spec)
    with _Only(48 * Q + 8 * Q // 4):         # 48 bytes a node hold the table, 6 more the exponents
        plan.set_basis(T, bl.BLAST_BASIS_FP64)
    C = plan.cl(rq, bl.BLAST_FP64)
    plan.close()
    assert np.all(ref > 0) and np.max(np.abs(C / ref - 1.0)) < 2 * (N + Rn + X + 100) * 2.0 ** -53

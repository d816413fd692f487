"""The batch-size and grid rules of the tensor-core and FP32 contractions at
their edges: cosmology tiles that repeat over the lane quadrants, a partial
last tile with CTAs of its own, passes as units, fewer tiles than epilogue
turns, FP32 groups of 4, 8 and 16 cosmologies and every R-node count a thread
can hold.  A cosmology's bits do not depend on any of it, so each result equals
the same request evaluated alone, and one of them is held to the FP64 path:
e_ij <= 1e-4 on the tensor cores (their bar), and for FP32, whose sums of N +
n_R / 32 + 5 + 3 + n_chi terms round each at 2^-24 and whose operands are rounded
once, (N + n_R + n_chi + 16) 2^-24 of the sum of the terms' magnitudes.
"""
import numpy as np
import pytest

import oracle as orc
from paper_2410_03632_gb300 import blast as bl
from paper_2410_03632_gb300 import synth
from tests.metrics import eij

pytestmark = pytest.mark.gpu


def _have_gpu():
    try:
        import torch
        return torch.cuda.is_available()
    except Exception:
        return False


if not _have_gpu():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("name,sel", [("tc", [4]), ("tc", None), ("tck", [2]), ("tck", None), ("tcg", [0, 5])])
def test_tensor_core_batches(name, sel):
    spec = synth.plan_spec(name)
    plan = bl.Plan(spec)
    plan.precompute(bl.BASIS_ALL)
    chi, R, _ = plan.nodes()
    rqs = [synth.config_request(name, chi, R, i % 7) for i in range(150)]
    alone = [plan.cl(rq, bl.BLAST_BF16S, ell_sel=sel) for rq in rqs[:7]]
    ref = plan.cl(rqs[1], bl.BLAST_FP64, ell_sel=sel)
    assert np.max(eij(alone[1], ref, spec.max_clust, spec.max_lens)) < 1e-4
    for n in (2, 32, 40, 64, 65, 130, 150):
        for i, C in enumerate(plan.cl_batch(rqs[:n], bl.BLAST_BF16S, [sel] * n)):
            np.testing.assert_array_equal(C, alone[i % 7], err_msg=f"{name} batch {n} request {i}")
    plan.close()


@pytest.mark.parametrize("X,Rn,N,sym", [(5, 10, 7, 0), (6, 64, 33, 0), (5, 66, 20, 1), (7, 130, 64, 0), (5, 258, 17, 0),
                                        (5, 512, 96, 0)])
def test_fp32_groups(X, Rn, N, sym):
    ng, ns = 3, 2
    spec = synth.PlanSpec(np.array([2, 40, 300], np.int32), X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 1, 257, ng, ns,
                          sym)
    g = orc.Grid(spec.ells, X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 257, 1, r_form=sym)
    rng = np.random.default_rng(Rn)
    T = rng.standard_normal((3, 3, N, X * Rn))
    plan = bl.Plan(spec)
    plan.set_basis(T, bl.BLAST_BASIS_FP32)
    rqs = []
    for i in range(18):
        a, b = (ng, ns) if i % 3 else (1 + i % ng, i % (ns + 1))
        k, P = synth.pk_table(rng.uniform(-2.5, -1.5), 0.05, rng.uniform(0, 6), 0.8)
        rqs.append(synth.Request(a, b, rng.random((a + b, X)), rng.random((a + b, X * Rn)), rng.random(X),
                                 rng.random(X * Rn), k, P))
    alone = [plan.cl(rq, bl.BLAST_FP32) for rq in rqs]
    for rq, C in zip(rqs[:3], alone):
        a = g.fit(rq.k_tab, rq.p_tab)
        args = (rq.n_clust, rq.n_lens, rq.kern_chi, rq.kern_Rchi, rq.growth_chi, rq.growth_Rchi)
        size = g.cl(np.abs(T), np.abs(a), *args)
        assert np.all(np.abs(C - g.cl(T, a, *args)) <= (N + Rn + X + 16) * 2.0 ** -24 * size)
    for n in (2, 4, 5, 8, 9, 16, 18):
        for C, ref in zip(plan.cl_batch(rqs[:n], bl.BLAST_FP32), alone):
            np.testing.assert_array_equal(C, ref)
    plan.close()

"""The bounded waits of the FP64 tensor-core contraction and of the basis
integrals, made to run out.

The test hook has two warps of the first CTA wait on a barrier that nothing
completes, with a short limit.  The kernel records its error word and leaves
once its copies and MMAs in flight are done.  A call with host outputs reports
it itself, a stream-ordered one (blast_cl_noalloc, device outputs) at the next
call on the plan; results after that are the ones from before.
"""
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


@pytest.fixture(scope="module")
def plan():
    p = bl.Plan(synth.plan_spec("tc"))
    p.precompute(bl.BLAST_BASIS_FP64)
    yield p
    p.close()


@pytest.mark.parametrize("item", [0, 3])
def test_host_outputs(plan, item):
    chi, R, _ = plan.nodes()
    rqs = [synth.config_request("tc", chi, R, i) for i in range(3)]
    ref = plan.cl_batch(rqs, bl.BLAST_FP64)
    assert bl.blast_test_trip_wait(plan.h, item) == bl.BLAST_OK
    with pytest.raises(bl.BlastError) as ei:
        plan.cl_batch(rqs, bl.BLAST_FP64)
    assert ei.value.status == bl.BLAST_ETIMEOUT
    for a, b in zip(plan.cl_batch(rqs, bl.BLAST_FP64), ref):
        np.testing.assert_array_equal(a, b)


def test_noalloc_reports_the_call_before(plan):
    import torch

    chi, R, _ = plan.nodes()
    rq = synth.config_request("tc", chi, R, 0)
    dev = {f: torch.from_numpy(np.ascontiguousarray(getattr(rq, f))).cuda()
           for f in ("kern_chi", "kern_Rchi", "growth_chi", "growth_Rchi", "k_tab", "p_tab")}
    r = plan.request(rq, device_arrays=dev)
    out = torch.empty((bl.blast_npairs(rq.n_clust, rq.n_lens), plan.L), dtype=torch.float64, device="cuda")

    def call():
        rc = bl.blast_cl_noalloc(plan.h, r, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return rc

    assert call() == bl.BLAST_OK
    ref = out.clone()
    assert bl.blast_test_trip_wait(plan.h, 2) == bl.BLAST_OK
    assert call() == bl.BLAST_OK          # enqueued; its wait runs out on the device
    assert call() == bl.BLAST_ETIMEOUT
    out.fill_(float("nan"))
    assert call() == bl.BLAST_OK
    assert torch.equal(out, ref)


def test_basis_build(plan):
    ref = plan.basis()
    chi, R, _ = plan.nodes()
    rq = synth.config_request("tc", chi, R, 0)
    for window in (0, 7):
        assert bl.blast_test_trip_wait(plan.h, window) == bl.BLAST_OK
        with pytest.raises(bl.BlastError) as ei:
            plan.precompute(bl.BLAST_BASIS_FP64)
        assert ei.value.status == bl.BLAST_ETIMEOUT
        with pytest.raises(bl.BlastError) as ei:
            plan.cl(rq, bl.BLAST_FP64)
        assert ei.value.status == bl.BLAST_ENOBASIS
        plan.precompute(bl.BLAST_BASIS_FP64)
        np.testing.assert_array_equal(plan.basis(), ref)


def test_basis_build_after_a_call_that_gave_up(plan):
    """The build succeeds, and the earlier call's failure is reported by the next evaluation."""
    import torch

    ref = plan.basis()
    chi, R, _ = plan.nodes()
    rq = synth.config_request("tc", chi, R, 0)
    want = plan.cl(rq, bl.BLAST_FP64)
    out = torch.empty(want.shape, dtype=torch.float64, device="cuda")
    assert bl.blast_test_trip_wait(plan.h, 0) == bl.BLAST_OK
    assert bl.blast_cl(plan.h, plan.request(rq), bl.BLAST_FP64, out.data_ptr(), 1, None) == bl.BLAST_OK
    torch.cuda.synchronize()
    plan.precompute(bl.BLAST_BASIS_FP64)
    np.testing.assert_array_equal(plan.basis(), ref)
    with pytest.raises(bl.BlastError) as ei:
        plan.cl(rq, bl.BLAST_FP64)
    assert ei.value.status == bl.BLAST_ETIMEOUT
    np.testing.assert_array_equal(plan.cl(rq, bl.BLAST_FP64), want)

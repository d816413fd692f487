"""FP32 batches of 16 + 16 tracers whose weights lie more than 2^31 floats apart (9
to 12 GB of weights), one for every group size and R-node count of the kernel.  A
cosmology's bits do not depend on its batch, so the first and the last two equal
the same requests evaluated alone."""
import types

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


@pytest.mark.parametrize("X,Rn,n", [(11700, 128, 16), (58600, 128, 4), (12600, 256, 8), (14700, 512, 4), (6300, 512, 8)])
def test_weights_further_apart_than_a_32_bit_offset(X, Rn, n):
    import torch

    ng, ns = 16, 16
    Q = X * Rn
    per = 3 * (ng + ns) * (X + Q)          # floats of work space a request
    assert (n - 1) * per > 2 ** 31
    plan = bl.Plan(synth.PlanSpec(np.array([2], np.int32), X, 40.0, 2400.0, Rn, 0.2, 1.8, 2, 1e-4, 1.0, 1, 17, ng, ns))
    gen = torch.Generator("cuda").manual_seed(3)

    def rand(*shape):
        return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=gen)

    plan.set_basis(rand(3, 1, 2, Q).cpu().numpy(), bl.BLAST_BASIS_FP32)
    kern = {"kern_chi": rand(ng + ns, X), "kern_Rchi": rand(ng + ns, Q)}
    k, P = synth.pk_table(-2.0, 0.05, 0.0, 0.8)
    dev = {"k_tab": torch.tensor(k, device="cuda"), "p_tab": torch.tensor(P, device="cuda")}
    rq = types.SimpleNamespace(n_clust=ng, n_lens=ns, k_tab=k)
    reqs = [plan.request(rq, device_arrays=dict(kern, growth_chi=rand(X), growth_Rchi=rand(Q), **dev)) for _ in range(n)]
    shape = (bl.blast_npairs(ng, ns), 1)
    outs = [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(n)]
    assert bl.blast_cl_batch(plan.h, reqs, bl.BLAST_FP32, [o.data_ptr() for o in outs], 1, None) == bl.BLAST_OK
    torch.cuda.synchronize()
    for i in (0, n - 2, n - 1):
        one = torch.empty(shape, dtype=torch.float64, device="cuda")
        assert bl.blast_cl(plan.h, reqs[i], bl.BLAST_FP32, one.data_ptr(), 1, None) == bl.BLAST_OK
        torch.cuda.synchronize()
        assert torch.equal(one, outs[i]) and bool(torch.all(one > 0))
    plan.close()

"""FP64 contraction on the tensor cores at the edges of its tiles.

Random bases with a wide spread of column and entry sizes, every spectrum
against the oracle's FP64 evaluation of the same table.  Both sides add at
most N + n_R + n_chi terms with a rounding each and share a fit good to a few
units in the last place of its largest coefficient, so a spectrum differs by
less than 1e-12 of the sum of its terms' magnitudes (with every coefficient at
its largest): (128 + 512 + 64) 2^-53 = 8e-14, plus 50 units for the fit.
A cosmology's bits do not depend on the batch.
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


def _setup(X, Rn, N, ng, ns, sym, seed=0, L=3):
    spec = synth.PlanSpec(np.array([2, 40, 300, 500][:L], np.int32), X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 1, 257,
                          ng, ns, sym)
    g = orc.Grid(spec.ells, X, 40.0, 2400.0, Rn, 0.2, 1.8, N, 1e-4, 1.0, 257, 1, r_form=sym)
    rng = np.random.default_rng(seed)
    T = rng.standard_normal((3, L, N, X * Rn)) * np.exp2(rng.integers(-40, 41, (3, L, 1, X * Rn)))
    T *= np.exp2(-rng.integers(0, 30, T.shape) * (rng.random(T.shape) < 0.3))
    T[:, :, :, 5::97] = 0.0          # empty columns
    T[:, :, :, 7::89] *= 2.0 ** -960  # columns too small to matter
    return spec, g, T


def _requests(plan, n, ng, ns, ragged, seed=1):
    chi, R, _ = plan.nodes()
    rng = np.random.default_rng(seed)
    out = []
    for i in range(n):
        a, b = (int(rng.integers(0, ng + 1)), int(rng.integers(1, ns + 1))) if ragged and ns else (ng, ns)
        Q = chi.size * R.size
        k, P = synth.pk_table(rng.uniform(-2.5, -1.5), 0.05, rng.uniform(0, 6), 0.8)
        out.append(synth.Request(a, b, rng.random((a + b, chi.size)), rng.random((a + b, Q)), rng.random(chi.size),
                                 rng.random(Q), k, P))
    return out


SHAPES = [
    # n_chi, n_R, n_cheb, clust, lens, r_form, batch, ragged
    (5, 2, 2, 1, 1, 0, 1, False),       # smallest: many chi nodes in a tile, one K step
    (13, 10, 7, 2, 0, 0, 2, False),     # twelve chi nodes a tile, one kind of tracer only
    (9, 64, 32, 1, 1, 0, 3, False),     # two chi nodes a tile
    (7, 66, 33, 3, 2, 0, 5, True),      # one chi node in part of a tile, a chunk and one order
    (6, 128, 64, 5, 5, 0, 16, False),   # full tile, full group
    (5, 130, 76, 5, 5, 0, 17, True),    # two R tiles; largest order of the unsigned digits; two groups
    (5, 192, 77, 10, 10, 0, 4, False),  # smallest order of the balanced digits
    (5, 384, 96, 16, 16, 0, 33, True),  # three R tiles, most tracers, three groups
    (5, 512, 128, 2, 3, 0, 2, False),   # largest n_R and order
    (7, 34, 20, 4, 3, 1, 6, True),      # symmetrised form: both kinds in one list
    (5, 160, 90, 16, 16, 1, 2, False),  # the same at 32 rows
]


@pytest.mark.parametrize("X,Rn,N,ng,ns,sym,n,ragged", SHAPES)
def test_against_oracle_and_alone(X, Rn, N, ng, ns, sym, n, ragged):
    spec, g, T = _setup(X, Rn, N, ng, ns, sym)
    plan = bl.Plan(spec)
    plan.set_basis(T, bl.BLAST_BASIS_FP64)
    rqs = _requests(plan, n, ng, ns, ragged)
    outs = plan.cl_batch(rqs, bl.BLAST_FP64)
    for i, (rq, C) in enumerate(zip(rqs, outs)):
        a = g.fit(rq.k_tab, rq.p_tab)
        args = (rq.n_clust, rq.n_lens, rq.kern_chi, rq.kern_Rchi, rq.growth_chi, rq.growth_Rchi)
        ref = g.cl(T, a, *args)
        size = g.cl(np.abs(T), np.full_like(a, np.abs(a).max()), *args)
        assert np.all(np.abs(C - ref) <= 1e-12 * size), float(np.max(np.abs(C - ref) / size))
        if i in (0, n - 1):
            np.testing.assert_array_equal(plan.cl(rq, bl.BLAST_FP64), C)
    plan.close()


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e-300])
def test_tables_the_digits_cannot_hold(bad):
    """An infinity, a NaN or a whole ell under 2^-700 keeps FP64's own arithmetic for the table."""
    spec, g, T = _setup(6, 32, 24, 2, 2, 0)
    if bad == 1e-300:
        T[1, 1] = bad * np.random.default_rng(2).standard_normal(T[1, 1].shape)
    else:
        T[1, 1, 3, 40] = bad
    plan = bl.Plan(spec)
    plan.set_basis(T, bl.BLAST_BASIS_FP64)
    rq = _requests(plan, 1, 2, 2, False)[0]
    C = plan.cl(rq, bl.BLAST_FP64)
    a = g.fit(rq.k_tab, rq.p_tab)
    args = (2, 2, rq.kern_chi, rq.kern_Rchi, rq.growth_chi, rq.growth_Rchi)
    if bad == 1e-300:
        ref = g.cl(T, a, *args)
        size = g.cl(np.abs(T), np.full_like(a, np.abs(a).max()), *args)
        assert np.all(np.abs(C - ref) <= 1e-12 * size) and np.all(C[3:7, 1] != 0.0)
    else:
        assert not np.any(np.isfinite(C[3:7, 1])) and np.all(np.isfinite(np.delete(C, 1, axis=1)))
    plan.close()


def test_coefficients_of_any_size():
    """P(k) scaled by powers of two scales the spectra exactly, down to the smallest normal coefficients."""
    spec, g, T = _setup(6, 32, 24, 2, 2, 0)
    T[:, :, :, 7::89] = 1.0
    plan = bl.Plan(spec)
    plan.set_basis(T, bl.BLAST_BASIS_FP64)
    rq = _requests(plan, 1, 2, 2, False)[0]
    p0 = rq.p_tab
    ref = plan.cl(rq, bl.BLAST_FP64)
    for e in (-900, -300, 300, 900):
        rq.p_tab = p0 * 2.0 ** e
        got = plan.cl(rq, bl.BLAST_FP64)
        # ln P rounds differently at another size: its error, |ln P| 2^-53 <= 640 2^-53, is P's relative one
        size = g.cl(np.abs(T), np.full(24, np.abs(g.fit(rq.k_tab, p0)).max()), 2, 2, rq.kern_chi, rq.kern_Rchi,
                    rq.growth_chi, rq.growth_Rchi)
        assert np.all(np.abs(got * 2.0 ** -e - ref) <= 1e-11 * size)
    plan.close()

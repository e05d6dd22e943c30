"""The persistent block solver in its cluster shapes: every block length and storage, an odd number of
right-hand sides, every launch shape (in FP64 also the one with eight lanes per site), against the oracle's block operator.

The bar is the solver's own target: the true residual of every right-hand side over the colour, by
the oracle's FP64 operator, at most tol_block (the defect correction stops there).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import core as oc
from paper_1211_1214_gb300 import binding, synth

pytestmark = pytest.mark.gpu

LATTICES = [((4, 4, 4, 8), 2), ((8, 8, 8, 16), 4), ((12, 12, 12, 12), 6), ((16, 16, 16, 16), 8)]


@pytest.mark.parametrize("dims,l", LATTICES, ids=["l2", "l4", "l6", "l8"])
def test_block_solver_cluster_shapes(dims, l):
    U = synth.gauge_field(dims, 0.25, seed=5)
    ctx = binding.Context(dims, (l,) * 4)
    ctx.load_gauge(U)
    ctx.set_params(1.3, 0.08, 0.06)
    lat = oc.Lattice(dims, (l,) * 4, U, 1.3)
    col = lat.colour()
    b = synth.spinor_field(dims, seed=6, nrhs=3)
    for prec, low16 in ((binding.FP64, False), (binding.MIXED_FP32, False), (binding.MIXED_FP16, True),
                        (binding.MIXED_BF16, True)):
        tol = 1e-13 if prec == binding.FP64 else 1e-12
        ctx.set_solver(prec, tol_outer=1e-10, tol_block=tol)
        ctx.set_low_precision(True, low16)
        for form in (0, 1, 2):
            ctx.block_config(form)
            for colour in (0, 1):
                x = np.zeros_like(b)
                ctx.solve_block(colour, 0.06, b, x, nrhs=3)
                for r in range(3):
                    bc = b[r].copy()
                    bc[col != colour] = 0
                    res = bc - lat.apply(0.06, x[r], rows=colour, cols=colour)
                    # the oracle's own rounding of D x is about 1e-15
                    assert np.linalg.norm(res) <= (tol + 2e-14) * np.linalg.norm(bc), (prec, form, colour, r)
                    assert np.max(np.abs(x[r][col != colour])) == 0.0
    # a zero right-hand side beside others converges at once and leaves zeros
    ctx.set_solver(binding.MIXED_FP32, tol_outer=1e-10, tol_block=1e-12)
    b[1] = 0
    x = np.ones_like(b)
    ctx.solve_block(0, 0.06, b, x, nrhs=3)
    assert np.max(np.abs(x[1])) == 0.0
    ctx.close()

"""The captured CG iteration of a context follows the shift of the call.

A context keeps the graph of its last solve. Solves without and with a shift take different
launches (the sum of |p|^2), on lattices of the eight-thread kernels (V/2 = 1080), on the last one
of them in FP64 but not in FP32 / FP16 storage (7296) and above (9800, a ragged last block)."""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(6, 6, 6, 10), (16, 6, 4, 38), (14, 14, 10, 10)])
@pytest.mark.parametrize("prec", ["double", "single", "half"])
def test_shift_changes_on_one_context(bq, dims, prec):  # noqa: F811
    lat, U, A, p = make(bq, dims, kappa=0.12, csw=1.0, mu=0.05, recon=18 if prec == "double" else 12, precision=prec)
    op = oracle.Operator(p, U, A)
    b = synth.gaussian_spinor(lat.Vh, 4)
    runs = {}
    for graphs in (True, False):
        bq.bq_set_cuda_graphs(lat.ctx, graphs)
        runs[graphs] = []
        for shift in (0.0, 0.3, 0.0, 0.05):
            x = np.empty_like(b)
            st = bq.bq_solve_cg(lat.ctx, x, b, tol=1e-10, precision=prec, shift=shift, max_iter=1000)
            assert rel(op.mdagm(x) + shift * x, b) < 1e-10
            runs[graphs].append((st["iterations"], x))
    for (n1, x1), (n2, x2) in zip(runs[True], runs[False]):
        assert n1 == n2 and np.array_equal(x1, x2)
    lat.close()

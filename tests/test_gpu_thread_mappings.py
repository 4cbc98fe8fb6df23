"""The hopping kernels that spread a site over eight threads (small lattices) or two
(FP64 units), and the one-thread kernels above them, against the FP64 oracle.

Sizes at the edges of the rules: a half-filled block of 16 sites (V/2 = 8), ragged
tails (V/2 mod 16 = 8), and lattices on both sides of the FP32 / FP16 (4864) and
FP64 (7296) limits. Tolerances per apply as everywhere: 1e-13, 1e-6, 5e-3.
"""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import TOL, bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu

# V/2 = 8, 1080 (tail 8), 4864 (the last FP32 / FP16 lattice of eight threads per site), 5000, 7296 (the last
# FP64 one), 9800 (tail 8)
DIMS = [(2, 2, 2, 2), (6, 6, 6, 10), (16, 4, 4, 38), (10, 10, 10, 10), (16, 6, 4, 38), (14, 14, 10, 10)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec,recon,charge", [("double", 18, 2.0 / 3.0), ("double", 12, 0.0), ("single", 18, -1.0 / 3.0),
                                               ("single", 12, 0.0), ("half", 12, 0.0)])
def test_applies(bq, dims, prec, recon, charge):  # noqa: F811
    lat, U, A, p = make(bq, dims, mu=0.1, charge=charge, recon=recon, precision=prec)
    op = oracle.Operator(p, U, A)
    psi = synth.gaussian_spinor(lat.Vh, 3)
    src, out = lat.pack(psi, prec), lat.spinor(prec)
    for par in (0, 1):
        for dag in (False, True):
            bq.bq_apply_dhop(lat.ctx, out, src, par, dag, prec)
            assert rel(lat.unpack(out, prec), oracle.dhop(p, U, A, psi, par, dag)) < TOL[prec], (par, dag)
    for dag in (False, True):
        bq.bq_apply_mhat(lat.ctx, out, src, dag, prec)
        assert rel(lat.unpack(out, prec), op.mhat(psi, dag)) < TOL[prec], dag
    bq.bq_apply_mdagm(lat.ctx, out, src, prec)
    assert rel(lat.unpack(out, prec), op.mdagm(psi)) < TOL[prec]
    lat.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 10), (16, 6, 4, 38)])
@pytest.mark.parametrize("prec", ["double", "single", "half"])
@pytest.mark.parametrize("shift", [0.0, 0.3])
def test_fused_cg(bq, dims, prec, shift):  # noqa: F811
    """CG with its vector work inside the eight-thread kernels: true residual, eager and captured alike."""
    lat, U, A, p = make(bq, dims, kappa=0.12, csw=1.0, mu=0.05, recon=18 if prec == "double" else 12, precision=prec)
    op = oracle.Operator(p, U, A)
    b = synth.gaussian_spinor(lat.Vh, 4)
    xs = []
    for graphs in (True, False):
        bq.bq_set_cuda_graphs(lat.ctx, graphs)
        x = np.empty_like(b)
        bq.bq_solve_cg(lat.ctx, x, b, tol=1e-10, precision=prec, shift=shift)
        assert rel(op.mdagm(x) + shift * x, b) < 1e-10
        xs.append(x)
    assert np.array_equal(xs[0], xs[1])
    lat.close()


def test_fp64_links_follow_the_storage_setting(bq):  # noqa: F811
    """12 reals of links that are not SU(3): the third row is conj(row 0 x row 1) in either FP64 arithmetic, and
    switching back to 18 brings the stored row back."""
    dims = (4, 4, 4, 4)
    lat, U, A, p = make(bq, dims)
    bad = U.copy()
    bad[:, :, 2] *= 1.5
    bq.bq_set_gauge(lat.ctx, bad)
    psi = synth.gaussian_spinor(lat.Vh, 5)
    src, out = lat.pack(psi), lat.spinor()
    for arith in ("native", "df64"):
        bq.bq_set_fp64_arith(lat.ctx, arith)
        for recon, links in ((18, bad), (12, U), (18, bad)):
            bq.bq_set_recon(lat.ctx, "double", recon)
            bq.bq_apply_dhop(lat.ctx, out, src, 0, False, "double")
            assert rel(lat.unpack(out), oracle.dhop(p, links, A, psi, 0, False)) < TOL["double"], (arith, recon)
    lat.close()


@pytest.mark.parametrize("prec", ["single", "half"])
@pytest.mark.parametrize("counts,expect", [((1, 1), -1), ((7,), -1), ((8,), None), ((15, 1), None), ((14, 1), -1)])
def test_default_batch_mapping(bq, prec, counts, expect):  # noqa: F811
    """The default of the batched apply: tiles from eight right-hand sides per lattice on average."""
    lats = [make(bq, d, recon=12, precision=prec, seed=i + 1) for i, d in enumerate([(6, 4, 6, 10), (4, 4, 4, 6)][:len(counts)])]
    ctxs, ins, outs, want = [], [], [], []
    for (lat, U, A, p), n in zip(lats, counts):
        op = oracle.Operator(p, U, A)
        for k in range(n):
            psi = synth.gaussian_spinor(lat.Vh, k)
            ctxs.append(lat)
            ins.append(lat.pack(psi, prec))
            outs.append(lat.spinor(prec))
            want.append(op.mdagm(psi))
    bq.bq_apply_mdagm_batch([c.ctx for c in ctxs], outs, ins, prec)
    assert bq.bq_get_batch_mapping(ctxs[0].ctx) == (expect or {"single": -3, "half": -4}[prec])
    for c, o, w in zip(ctxs, outs, want):
        assert rel(c.unpack(o, prec), w) < TOL[prec]
    for lat, *_ in lats:
        lat.close()

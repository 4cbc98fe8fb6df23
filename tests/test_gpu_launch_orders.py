"""Launches that run backwards, streaming loads and the one-thread CG steps, on lattices with ragged last blocks.

A x - k D launches run from the last site to the first, and FP32 links and clover blocks pass L1 by, only
where the working set exceeds L2 (129 MB): the lattices here are just beyond that for their storage, and none
of their V/2 is a multiple of a block's sites. Everything against the FP64 oracle, tolerances per apply as
everywhere."""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import TOL, bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu


# V/2 = 113 256: backwards with either link storage, streaming with 18-real links; 149 072: streaming with 12;
# 192 192: backwards in FP16 storage; 49 896: backwards in both FP64 arithmetics (blocks of 16 and 64 sites)
@pytest.mark.parametrize("dims,prec,arith,recon,charge", [
    ((22, 18, 22, 26), "single", "native", 18, 2.0 / 3.0), ((22, 18, 22, 26), "single", "native", 12, 0.0),
    ((22, 18, 22, 26), "single", "native", 8, 0.0), ((22, 22, 22, 28), "single", "native", 12, 0.0),
    ((24, 22, 26, 28), "half", "native", 12, 0.0), ((14, 18, 18, 22), "double", "native", 18, -1.0 / 3.0),
    ((14, 18, 18, 22), "double", "df64", 12, 0.0)])
def test_backward_and_streaming_applies(bq, dims, prec, arith, recon, charge):  # noqa: F811
    lat, U, A, p = make(bq, dims, mu=0.1, charge=charge, recon=recon, precision=prec)
    bq.bq_set_fp64_arith(lat.ctx, arith)
    op = oracle.Operator(p, U, A)
    psi = synth.gaussian_spinor(lat.Vh, 3)
    src, out = lat.pack(psi, prec), lat.spinor(prec)
    for dag in (False, True):
        bq.bq_apply_mhat(lat.ctx, out, src, dag, prec)
        assert rel(lat.unpack(out, prec), op.mhat(psi, dag)) < TOL[prec], dag
    bq.bq_apply_mdagm(lat.ctx, out, src, prec)
    assert rel(lat.unpack(out, prec), op.mdagm(psi)) < TOL[prec]
    lat.close()


@pytest.fixture(scope="module")
def two_lattices():
    """V/2 = 78 408 (backwards from two right-hand sides a unit in FP32, from eight in FP16) and 720 (forwards),
    with sources and Mhat^dag Mhat of them."""
    made = []
    for dims, n in (((22, 18, 18, 22), 8), ((6, 4, 6, 10), 2)):
        U = synth.gauge_field(dims, 0.2, 1)
        op = oracle.Operator(oracle.params(dims, kappa=0.12, csw=1.0, mu=0.05, t_bc=-1.0, charge=0.0), U)
        psis = [synth.gaussian_spinor(int(np.prod(dims)) // 2, k) for k in range(n)]
        made.append((dims, U, op, psis, [op.mdagm(v) for v in psis]))
    return made


def contexts(bq, two_lattices, prec):  # noqa: F811
    lats = []
    for dims, U, *_ in two_lattices:
        lat = bq.Lattice(dims, 0.12, 1.0, 0.05, -1.0, 0.0)
        bq.bq_set_recon(lat.ctx, prec, 12)
        bq.bq_set_gauge(lat.ctx, U)
        lats.append(lat)
    return lats


@pytest.mark.parametrize("prec", ["single", "half"])
@pytest.mark.parametrize("mapping", [-1, -2, -3, 2, 4, 8])
def test_backward_batches_of_two_lattices(bq, two_lattices, prec, mapping):  # noqa: F811
    lats = contexts(bq, two_lattices, prec)
    bq.bq_set_batch_mapping(lats[0].ctx, mapping)
    ctxs, ins, want = [], [], []
    for lat, (_, _, _, psis, res) in zip(lats, two_lattices):
        ctxs += [lat] * len(psis)
        ins += [lat.pack(v, prec) for v in psis]
        want += res
    outs = [c.spinor(prec) for c in ctxs]
    bq.bq_apply_mdagm_batch([c.ctx for c in ctxs], outs, ins, prec)
    for c, o, w in zip(ctxs, outs, want):
        assert rel(c.unpack(o, prec), w) < TOL[prec]
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("prec", ["single", "half"])
@pytest.mark.parametrize("shift", [0.0, 0.1])
def test_backward_fused_batch_cg(bq, two_lattices, prec, shift):  # noqa: F811
    """Block-interleaved batches run the vector work of CG inside the hopping launches: the counters hold its
    bytes with those of the A x - k D steps."""
    lats = contexts(bq, two_lattices, prec)
    bq.bq_set_batch_mapping(lats[0].ctx, -1)
    ctxs = [lats[0]] * 8 + [lats[1]] * 2
    ops = [two_lattices[0][2]] * 8 + [two_lattices[1][2]] * 2
    bs = two_lattices[0][3] + two_lattices[1][3]
    xs = [np.empty_like(b) for b in bs]
    bq.bq_reset_counters(lats[0].ctx)
    stats = bq.bq_solve_cg_batch([c.ctx for c in ctxs], xs, bs, tol=1e-8, precision=prec, shift=shift, delta=1e-2)
    assert bq.bq_get_counters(lats[0].ctx)["fused_bytes"][1 if prec == "single" else 2][2] > 0
    for op, b, x, st in zip(ops, bs, xs, stats):
        assert st["converged"] and rel(op.mdagm(x) + shift * x, b) < 1e-8
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("prec", ["single", "half"])
@pytest.mark.parametrize("recon", [8, 12, 18])
@pytest.mark.parametrize("shift", [0.0, 0.3])
def test_fused_cg_with_a_ragged_block(bq, prec, recon, shift):  # noqa: F811
    """V/2 = 9800 (a last block of 72 sites) is beyond the eight-thread kernels."""
    lat, U, A, p = make(bq, (14, 14, 10, 10), kappa=0.12, csw=1.0, mu=0.05, recon=recon, precision=prec)
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

"""An operator launch that follows its fields' packing at once reads what was packed.

The packing is queued by a batched call that is refused for its second system; before the next launch on
that stream another context on another stream runs, and another thread makes the call. Every result equals
that of a context whose fields have long been packed, bit for bit."""
import threading

import numpy as np
import pytest

from paper_1711_03836_gb300 import synth
from test_gpu_parity import bq  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (16, 16, 16, 16)])
@pytest.mark.parametrize("prec", ["single", "half", "double"])
def test_launch_after_a_refused_batch(bq, dims, prec):  # noqa: F811
    import torch

    streams = [torch.cuda.Stream() for _ in range(2)]
    lat, other = [bq.Lattice(dims, 0.13, 1.5, 0.0, -1.0, 0.0, stream=s.cuda_stream) for s in streams]
    odd = bq.Lattice((4, 4, 4, 4), 0.13, 1.5, 0.0, -1.0, 0.0, stream=streams[0].cuda_stream)
    Us = [synth.gauge_field(dims, 0.3, seed) for seed in (1, 2)]
    Us = Us + [Us[0]]
    psi = synth.gaussian_spinor(lat.Vh, 3)
    src, out, oout = lat.pack(psi, prec), lat.spinor(prec), lat.spinor(prec)
    bq.bq_set_gauge(odd.ctx, synth.gauge_field((4, 4, 4, 4), 0.3, 1))
    bq.bq_set_recon(odd.ctx, prec, 12)  # not lat's storage: the batch is refused after lat's fields are packed
    osrc, od = odd.spinor(prec), odd.spinor(prec)
    for U in Us:
        for l in (lat, other):
            bq.bq_set_gauge(l.ctx, U)
        torch.cuda.synchronize()
        bq.bq_apply_mdagm(other.ctx, oout, src, prec)
        torch.cuda.synchronize()
        want = other.unpack(oout, prec)
        bq.bq_build_clover(lat.ctx)
        with pytest.raises(bq.BqError):
            bq.bq_apply_mdagm_batch([lat.ctx, odd.ctx], [out, od], [src, osrc], prec)
        bq.bq_apply_mdagm(other.ctx, oout, src, prec)
        t = threading.Thread(target=lambda: bq.bq_apply_mdagm(lat.ctx, out, src, prec))
        t.start()
        t.join()
        torch.cuda.synchronize()
        assert np.array_equal(lat.unpack(out, prec), want)
    for l in (lat, other, odd):
        l.close()


@pytest.mark.parametrize("arith", ["df64", "native"])
def test_batch_of_two_streams_fp64(bq, arith):  # noqa: F811
    """The FP64 fields of a batch whose second system lives on another stream, in either FP64 arithmetic: the
    batched operator and solve right after new links, against the same calls one context at a time."""
    import torch

    dims = [(8, 8, 8, 8), (16, 16, 16, 16)]
    lats = [bq.Lattice(d, 0.12, 1.0, 0.0, -1.0, 0.0, stream=torch.cuda.Stream().cuda_stream) for d in dims]
    for l in lats:
        bq.bq_set_fp64_arith(l.ctx, arith)
    psis = [synth.gaussian_spinor(l.Vh, 3) for l in lats]
    src, out, one = [[l.pack(v) if k == 0 else l.spinor() for l, v in zip(lats, psis)] for k in range(3)]
    for seed in (1, 2, 1):
        Us = [synth.gauge_field(d, 0.3, seed) for d in dims]
        for l, U in zip(lats, Us):
            bq.bq_set_gauge(l.ctx, U)
            bq.bq_build_clover(l.ctx)
        torch.cuda.synchronize()
        bq.bq_apply_mdagm_batch([l.ctx for l in lats], out, src, "double")
        torch.cuda.synchronize()
        got = [l.unpack(o) for l, o in zip(lats, out)]
        xs = [np.empty_like(v) for v in psis]
        bq.bq_solve_cg_batch([l.ctx for l in lats], xs, psis, tol=1e-10, precision="single")
        for l, s, o, g, x, v in zip(lats, src, one, got, xs, psis):
            bq.bq_apply_mdagm(l.ctx, o, s, "double")
            torch.cuda.synchronize()
            want = l.unpack(o)
            assert np.linalg.norm(g - want) <= 1e-13 * np.linalg.norm(want)
            y = l.pack(x)
            bq.bq_apply_mdagm(l.ctx, o, y, "double")
            torch.cuda.synchronize()
            assert np.linalg.norm(l.unpack(o) - v) <= 1.01e-10 * np.linalg.norm(v)
    for l in lats:
        l.close()

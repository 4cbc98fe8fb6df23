"""A configuration is prepared in the memory of the context's own fields.

Once a context has run, its next configuration (links, clover, log det, stout links, first operator) takes no
further device memory, and it goes through with less memory free than one more copy of the links would need.
The links are then read through a buffer in pieces, and the split links lie in fields that are out of date, in
the memory that takes the result, in memory allocated for the call, or links are split at each use: every way
gives the same bits."""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu

ORDERS = {  # which fields are out of date when the stout step runs
    "stout first": ("hop", "clover", "op"),
    "clover first": ("clover", "hop", "op"),
    "operator only": ("op", "hop", "clover"),
    "links only": ("hop", "hop", "hop"),
}


def one_pass(bq, lat, U, order, prec, src, out, hop):
    bq.bq_set_gauge(lat.ctx, U)
    for step in order:
        if step == "hop":
            bq.bq_get_hop_links(lat.ctx, hop)
        elif step == "clover":
            bq.bq_build_clover(lat.ctx)
            bq.bq_clover_logdet(lat.ctx, 1)
        else:
            bq.bq_apply_mdagm(lat.ctx, out, src, prec)


@pytest.mark.parametrize("order", list(ORDERS))
@pytest.mark.parametrize("prec,arith,n_iter", [("single", "native", 1), ("half", "native", 2), ("double", "native", 1),
                                               ("double", "df64", 3)])
def test_every_place_of_the_split_links(bq, order, prec, arith, n_iter):  # noqa: F811
    """Two configurations in turn on one context, against a fresh context and the oracle."""
    dims = (6, 6, 6, 6)
    lat, U, A, p = make(bq, dims, mu=0.1, recon=12, precision=prec)
    bq.bq_set_fp64_arith(lat.ctx, arith)
    bq.bq_set_stout(lat.ctx, 0.1, n_iter)
    Us = [U, synth.gauge_field(dims, 0.3, 9)]
    psi = synth.gaussian_spinor(lat.Vh, 3)
    src, out = lat.pack(psi, prec), lat.spinor(prec)
    hops = []
    for k in (0, 1, 0, 1):
        hop = np.empty_like(U)
        one_pass(bq, lat, Us[k], ORDERS[order], prec, src, out, hop)
        assert rel(hop, oracle.stout(dims, Us[k], 0.1, n_iter)) < 1e-13
        if "op" in ORDERS[order]:
            fresh = make(bq, dims, mu=0.1, recon=12, precision=prec)[0]
            bq.bq_set_fp64_arith(fresh.ctx, arith)
            bq.bq_set_stout(fresh.ctx, 0.1, n_iter)
            bq.bq_set_gauge(fresh.ctx, Us[k])
            ref = fresh.spinor(prec)
            bq.bq_apply_mdagm(fresh.ctx, ref, src, prec)
            assert np.array_equal(lat.unpack(out, prec), fresh.unpack(ref, prec))
            fresh.close()
        hops.append(hop)
    assert np.array_equal(hops[0], hops[2]) and np.array_equal(hops[1], hops[3])
    lat.close()


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("order", ["clover first", "operator only"])
def test_next_configuration_needs_no_memory(bq, where, order):  # noqa: F811
    import torch

    dims = (32, 32, 32, 32)  # 604 MB of links
    U = torch.eye(3, dtype=torch.complex128, device="cuda").repeat(int(np.prod(dims)), 4, 1, 1)
    hop = torch.empty_like(U) if where == "device" else np.empty(tuple(U.shape), np.complex128)
    if where == "host":
        U = U.cpu().numpy()
    lat = bq.Lattice(dims, 0.13, 1.0, 0.0, -1.0, 0.0)
    bq.bq_set_recon(lat.ctx, "single", 12)
    bq.bq_set_stout(lat.ctx, 0.1, 1)
    src, out = lat.pack(synth.gaussian_spinor(lat.Vh, 3), "single"), lat.spinor("single")
    one_pass(bq, lat, U, ORDERS[order], "single", src, out, hop)
    want = lat.unpack(out, "single")
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    one_pass(bq, lat, U, ORDERS[order], "single", src, out, hop)
    assert torch.cuda.mem_get_info()[0] >= free - (16 << 20)  # one more copy of the links is 604 MB
    fill = torch.empty(free - (350 << 20), dtype=torch.uint8, device="cuda")
    one_pass(bq, lat, U, ORDERS[order], "single", src, out, hop)
    del fill
    torch.cuda.empty_cache()
    assert np.array_equal(lat.unpack(out, "single"), want)
    lat.close()

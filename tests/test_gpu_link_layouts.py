"""The library's own link order, the split links and the exponential of the stout step.

V = 1296 leaves half a block of 32 sites; host and device links must come back
bit for bit; the stout step takes its three branches of exp(X) (series to order
11, to order 18, closed form) at small, moderate and large rho on smooth and
rough links. Tolerance 1e-13 as for every FP64 field."""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 6), (4, 4, 4, 4)])
def test_links_come_back_unchanged(bq, dims):  # noqa: F811
    import torch

    lat, U, A, p = make(bq, dims)
    dev = torch.from_numpy(U.copy()).cuda()
    for src in (U, dev):
        bq.bq_set_gauge(lat.ctx, src)
        back, dback = np.empty_like(U), torch.empty_like(dev)
        bq.bq_build_clover(lat.ctx)  # uses the work field that stages host links
        bq.bq_get_hop_links(lat.ctx, back)
        bq.bq_get_hop_links(lat.ctx, dback)
        assert np.array_equal(back, U) and torch.equal(dback, dev)
    lat.close()


@pytest.mark.parametrize("dims", [(6, 6, 6, 6), (2, 4, 2, 6)])
@pytest.mark.parametrize("eps", [0.05, 0.3, 2.0])
@pytest.mark.parametrize("rho,n_iter", [(0.05, 1), (0.1, 3), (0.4, 2), (1.0, 1)])
def test_stout_branches(bq, dims, eps, rho, n_iter):  # noqa: F811
    lat, U, A, p = make(bq, dims, eps=eps)
    bq.bq_build_clover(lat.ctx)
    bq.bq_set_stout(lat.ctx, rho, n_iter)
    got = bq.bq_get_hop_links(lat.ctx, np.empty_like(U))
    want = oracle.stout(dims, U, rho, n_iter)
    assert rel(got, want) < 1e-13
    lat.close()

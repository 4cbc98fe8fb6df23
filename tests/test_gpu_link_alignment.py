"""Links in device memory that lie on no 16-byte boundary: a slice of a larger allocation.

8 bytes off (doubles, but no pairs of doubles) and 4 bytes off (no double at all: through a copy); V = 1296
leaves half a block of 32 sites. The links come back bit for bit and the memory around them stays as it was."""
import numpy as np
import pytest

from test_gpu_parity import bq, make  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 6)])
@pytest.mark.parametrize("offset", [0, 8, 4])
def test_links_at_any_alignment(bq, dims, offset):  # noqa: F811
    import torch

    lat, U, A, p = make(bq, dims)
    raw = torch.from_numpy(U.copy().view(np.uint8).reshape(-1)).cuda()
    n = raw.numel()
    src = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")
    src[offset:offset + n] = raw
    dst = torch.full((n + 32,), 7, dtype=torch.uint8, device="cuda")
    bq.bq_set_gauge(lat.ctx, make(bq, dims, seed=9)[1])
    bq.bq_set_gauge(lat.ctx, src[offset:offset + n])
    bq.bq_get_hop_links(lat.ctx, dst[offset:offset + n])
    assert torch.equal(dst[offset:offset + n], raw)
    assert bool((dst[:offset] == 7).all()) and bool((dst[offset + n:] == 7).all())
    back = np.empty_like(U)
    bq.bq_get_hop_links(lat.ctx, back)
    assert np.array_equal(back, U)
    lat.close()

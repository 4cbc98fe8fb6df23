"""Double-float links follow the storage setting of FP64 links, and outlast a setting that comes and goes."""
import numpy as np
import pytest

import oracle
from paper_1711_03836_gb300 import synth
from test_gpu_parity import TOL, bq, make, rel  # noqa: F401

pytestmark = pytest.mark.gpu


def test_setting_forth_and_back_packs_nothing(bq):  # noqa: F811
    lat, U, A, p = make(bq, (4, 4, 4, 4))
    bad = U.copy()
    bad[:, :, 2] *= 1.5  # not SU(3): 12 and 18 reals are different operators
    bq.bq_set_gauge(lat.ctx, bad)
    bq.bq_set_fp64_arith(lat.ctx, "df64")
    psi = synth.gaussian_spinor(lat.Vh, 5)
    src, out = lat.pack(psi), lat.spinor()
    want = {r: oracle.dhop(p, u, A, psi, 0, False) for r, u in ((18, bad), (12, U))}
    packed = []
    for settings in ((18,), (12, 18), (12,), (18, 12), (12, 18)):
        for r in settings:
            bq.bq_set_recon(lat.ctx, "double", r)
        bq.bq_reset_counters(lat.ctx)
        bq.bq_apply_dhop(lat.ctx, out, src, 0, False, "double")
        packed.append(bq.bq_get_counters(lat.ctx)["launches"] > 1)
        assert rel(lat.unpack(out), want[settings[-1]]) < TOL["double"], settings
    assert packed == [True, False, True, False, True]
    lat.close()

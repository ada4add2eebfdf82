"""What a plan reports as its launch configuration, and what an autotuned plan may take over from an
earlier one."""
import math

import pytest
import torch

from paper_2203_15963_gb300 import native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu
FREQ = 230e9


@pytest.fixture(scope="module")
def torus():
    native.build()
    native.load()
    gp = S.grid_params_for(32, 16, 16)
    return gp, torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()


@pytest.mark.parametrize("precision", [native.BL_PREC_FP64, native.BL_PREC_MIXED,
                                       native.BL_PREC_FAST])
def test_adaptive_plan_reports_the_defaults(torus, precision):
    gp, prim = torus
    cam = S.Camera(theta=math.radians(60.0), n=16)
    met = S.Metric(spin=0.9, precision=precision)
    dt = torch.float64 if precision == native.BL_PREC_FP64 else torch.float32
    out = {"stokes": torch.empty((4, 32, 32), dtype=dt, device="cuda")}
    ad = native.adapt_struct(8, 1, native.BL_CRIT_REL_GRAD, 0.1, 5)
    plan = native.AdaptivePlan([cam], [met], [gp], [prim], [FREQ], ad, [out])
    cfg = plan.config()
    plain = native.Plan([cam], [met], [gp], [prim], [FREQ],
                        [{"stokes": torch.empty((4, 16, 16), dtype=dt, device="cuda")}])
    assert cfg == plain.config()
    assert cfg["geo_ctas_per_sm"] >= 1 and cfg["tr_ctas_per_sm"] >= 1 and cfg["ilv_block"] == 0
    plan.run()
    plan.check()
    plan.close()
    plain.close()

"""Cameras so far out that the metric's f underflows to zero in the integrator's arithmetic: the ray
is straight, as in flat space."""
import math

import pytest
import torch

from paper_2203_15963_gb300 import native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [native.BL_PREC_FP64, native.BL_PREC_MIXED])
@pytest.mark.parametrize("integrator", [native.BL_INT_DP, native.BL_INT_RK4])
@pytest.mark.parametrize("r", [1e30, 1e50, 1e52, 1e60])
def test_far_rays_are_straight(precision, integrator, r):
    """Impact parameters of 0.18 r and more: deflections are below 1e-28, rounding some 1e-16 an
    evaluation, so 1e-12 of the largest component after at most some hundred steps."""
    native.build()
    native.load()
    cam = S.Camera(theta=math.radians(60.0), n=4, r=r, width=r)
    ends = []
    for flat in (0, 1):
        met = S.Metric(spin=0.9, precision=precision, flat=flat, integrator=integrator, f_step=0.05)
        out = {"end_state": torch.empty((4, 4, 8), dtype=torch.float64, device="cuda"),
               "status": torch.empty((4, 4), dtype=torch.int32, device="cuda")}
        native.blacklight_geodesics(cam, met, out)
        assert native.RAY_STATUS[int(out["status"].min())] == "escaped"
        assert native.RAY_STATUS[int(out["status"].max())] == "escaped"
        ends.append(out["end_state"])
    for part in (slice(1, 4), slice(4, 8)):   # position, momentum
        a, b = ends[0][..., part], ends[1][..., part]
        if part.start == 1:   # (a fixed-step ray stops at its own step's end: across the ray only)
            k = ends[1][..., 5:8]
            k = k / k.norm(dim=-1, keepdim=True)
            a, b = (v - (v * k).sum(-1, keepdim=True) * k for v in (a, b))
        assert float((a - b).abs().max()) <= 1e-12 * float(ends[1][..., part].abs().max())

"""The FP64-arithmetic kernels: every launch shape traces a ray with the same bits,
and the FP32 decision into how many samples a step splits (FP64 where its error bound straddles
a boundary) gives the FP64 decision, which a trace with auxiliary images always takes."""
import math

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu
FREQ = 230e9


@pytest.fixture(scope="module")
def torus():
    native.build()
    native.load()
    gp = S.grid_params_for(64, 32, 32)
    return gp, {a: torch.from_numpy(S.make_torus(gp, a, S.BASE_SEED)).cuda() for a in (0.0, 0.97)}


def _outs(n, precision, aux=False):
    dt = torch.float64 if precision == native.BL_PREC_FP64 else torch.float32
    return images.alloc_outputs(n, dt, end_state=True, samples=True, aux=aux)


def _image(n, spin, inc, precision, **metric):
    return (S.Camera(theta=math.radians(inc), n=n),
            S.Metric(spin=spin, precision=precision, **metric))


@pytest.mark.parametrize("n,spin,inc,precision", [
    (1, 0.97, 60.0, native.BL_PREC_FP64), (37, 0.97, 80.0, native.BL_PREC_FP64),
    (48, 0.0, 17.0, native.BL_PREC_FP64), (37, 0.97, 80.0, native.BL_PREC_MIXED)])
def test_launch_shapes_give_the_same_bits(torus, n, spin, inc, precision):
    """The default shape against a plan with a set number of CTAs an SM (FP64: the 64-warp
    kernels)."""
    gp, prims = torus
    cam, met = _image(n, spin, inc, precision)
    a, b = _outs(n, precision), _outs(n, precision)
    images.trace_images([cam], [met], [gp], [prims[spin]], [FREQ], outs=[a])
    plan = native.Plan([cam], [met], [gp], [prims[spin]], [FREQ], [b],
                       config={"geo_ctas_per_sm": 2, "tr_ctas_per_sm": 2})
    plan.run()
    plan.check()
    plan.close()
    for k in a:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("precision", [native.BL_PREC_FP64, native.BL_PREC_MIXED])
def test_two_ctas_an_sm_give_the_same_bits(torus, precision):
    """592 rays an SM: between the waves that one CTA an SM serves and those that all do."""
    gp, prims = torus
    cam, met = _image(300, 0.97, 60.0, precision)
    a, b = _outs(300, precision), _outs(300, precision)
    images.trace_images([cam], [met], [gp], [prims[0.97]], [FREQ], outs=[a])
    plan = native.Plan([cam], [met], [gp], [prims[0.97]], [FREQ], [b],
                       config={"geo_ctas_per_sm": 1, "tr_ctas_per_sm": 1})
    plan.run()
    plan.check()
    plan.close()
    for k in a:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("spin,inc,ds_max,r_in", [
    (0.97, 5.0, 0.5, 1.01), (0.97, 88.0, 0.5, 1.0001), (0.0, 45.0, 0.3, 1.01),
    (0.97, 60.0, 2.0, 1.3), (0.97, 60.0, 40.0, 1.01)])
@pytest.mark.parametrize("precision", [native.BL_PREC_FP64, native.BL_PREC_MIXED])
def test_step_splitting_matches_the_fp64_decision(torus, spin, inc, ds_max, r_in, precision):
    gp, prims = torus
    n = 64
    cam, met = _image(n, spin, inc, precision, ds_max=ds_max, r_in_over_rhor=r_in)
    a, b = _outs(n, precision), _outs(n, precision, aux=True)
    images.trace_images([cam], [met], [gp], [prims[spin]], [FREQ], outs=[a])
    images.trace_images([cam], [met], [gp], [prims[spin]], [FREQ], outs=[b])
    for k in ("samples", "steps", "status", "end_state"):
        assert torch.equal(a[k], b[k]), k

"""What a plan reports as its launch configuration, and what an autotuned plan may take over from an
earlier one."""
import ctypes as C
import dataclasses
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


def _tuned(gp, prim, n=16, unpolarized=False, layout="planes", snapshots=1, autotune=True, **metric):
    """An FP64 plan (native.Plan has no flags)."""
    if snapshots > 1:
        gp = dataclasses.replace(gp, n_snapshots=snapshots, time_interp=1, t_first=0.0,
                                 dt_snapshots=40.0, t_camera=1035.0)
        prim = torch.stack([prim] * snapshots).contiguous()
    if layout == "cells":
        prim, gp = images.pack_grid(prim, gp)
    out = images.alloc_outputs(n, torch.float64)
    cam = S.Camera(theta=math.radians(60.0), n=n)
    met = S.Metric(spin=0.9, precision=native.BL_PREC_FP64, **metric)
    structs = (native.camera_struct(cam), native.metric_struct(met),
               native.grid_struct(gp, prim.data_ptr()), C.c_double(FREQ), native.out_struct(**out))
    flags = (native.BL_PLAN_AUTOTUNE if autotune else 0) | (native.BL_UNPOLARIZED if unpolarized else 0)
    plan = native.Plan.__new__(native.Plan)
    plan._h, plan._keep = C.c_void_p(), (prim, out)
    native._check(native.load().blacklight_plan_create(
        1, *(C.byref(v) for v in structs), None, flags, native._stream(None), C.byref(plan._h)))
    return plan


@pytest.mark.parametrize("other", [
    dict(unpolarized=True), dict(layout="cells"), dict(snapshots=2), dict(n=17),
    dict(integrator=native.BL_INT_RK4, f_step=0.05), "grid"], ids=str)
def test_autotuned_choice_is_not_taken_from_another_workload(torus, other):
    """A choice comes from the cache with the time it was made at, to the last bit; a plan that
    tunes for itself has a time of its own."""
    gp, prim = torus
    if other == "grid":
        gp2 = S.grid_params_for(32, 16, 20)
        first = _tuned(gp2, torch.from_numpy(S.make_torus(gp2, 0.9, S.BASE_SEED)).cuda())
    else:
        first = _tuned(gp, prim, **other)
    second, again = _tuned(gp, prim), _tuned(gp, prim)
    assert second.config()["run_ms"] != first.config()["run_ms"]
    assert again.config() == second.config()
    for p in (first, second, again):
        p.run()
        assert p.check() >= 0
        p.close()


def test_fixed_step_plan_reports_its_own_kernel(torus):
    """The RK kernel holds 3 CTAs an SM, the dense FP64 Dormand-Prince kernel 16."""
    gp, prim = torus
    dp = _tuned(gp, prim, autotune=False)
    rk = _tuned(gp, prim, autotune=False, integrator=native.BL_INT_RK4, f_step=0.05)
    assert 1 <= rk.config()["geo_ctas_per_sm"] < dp.config()["geo_ctas_per_sm"]
    dp.close()
    rk.close()


@pytest.mark.parametrize("precision", [native.BL_PREC_FP64, native.BL_PREC_MIXED])
@pytest.mark.parametrize("integrator,n", [(native.BL_INT_RK4, 37), (native.BL_INT_RK2, 37),
                                          (native.BL_INT_RK4, 300)])
@pytest.mark.parametrize("ctas", [1, 2])
def test_fixed_step_launch_shapes_give_the_same_bits(torus, precision, integrator, n, ctas):
    """The kernel's own rule (9 rays an SM: one CTA of an SM stays; 592: two) against a set number."""
    gp, prim = torus
    cam = S.Camera(theta=math.radians(80.0), n=n)
    met = S.Metric(spin=0.9, precision=precision, integrator=integrator, f_step=0.05)
    dt = torch.float64 if precision == native.BL_PREC_FP64 else torch.float32
    a, b = (images.alloc_outputs(n, dt, end_state=True, samples=True) for _ in range(2))
    images.trace_images([cam], [met], [gp], [prim], [FREQ], outs=[a])
    plan = native.Plan([cam], [met], [gp], [prim], [FREQ], [b],
                       config={"geo_ctas_per_sm": ctas, "tr_ctas_per_sm": ctas})
    assert plan.config()["geo_ctas_per_sm"] == ctas
    plan.run()
    plan.check()
    plan.close()
    for k in a:
        assert torch.equal(a[k], b[k]), k

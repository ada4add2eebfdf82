"""The learned form's work list: images whose samples all, partly or never reach the model, odd
sizes, several waves, both grid layouts and slow light, against the exact-fit transfer with a model
that reproduces nothing (so any row mix-up shows) and against itself in other launch splits."""
import dataclasses
import math

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu
FREQ = 230e9


@pytest.fixture(scope="module")
def data():
    native.build()
    native.load()
    gp = S.grid_params_for(64, 32, 32)
    prim = torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()
    params = torch.empty(native.MLP_PARAMS, dtype=torch.float32, device="cuda")
    native.blacklight_mlp_init(params, 5)
    return gp, prim, params


def _trace(gp, prim, n, workspace=None, coef=None):
    cam = S.Camera(theta=math.radians(60.0), n=n)
    met = S.Metric(spin=0.9, precision=native.BL_PREC_FAST)
    out = images.alloc_outputs(n, torch.float32)
    images.trace_images([cam], [met], [gp], [prim], [FREQ], outs=[out], workspace=workspace,
                        coef_mlp=coef)
    torch.cuda.synchronize()
    return out["stokes"]


@pytest.mark.parametrize("n", [1, 7, 33, 64])
@pytest.mark.parametrize("layout", ["planes", "cells"])
def test_waves_and_layouts_agree(data, n, layout):
    """Each row's outputs do not depend on its place in the list: one wave, many waves (a
    workspace that holds about 40 rays) and both layouts give the same bits."""
    gp, prim, params = data
    ref = _trace(gp, prim, n, coef=params)
    if layout == "cells":
        prim, gp = images.pack_grid(prim, gp)
    small = torch.empty(3 << 20, dtype=torch.uint8, device="cuda")
    assert torch.equal(_trace(gp, prim, n, coef=params), ref)
    assert torch.equal(_trace(gp, prim, n, workspace=small, coef=params), ref)
    if n > 7:
        assert float(ref[0].max()) > 0.0


def test_no_sample_in_the_domain_is_the_exact_image(data):
    """Plasma far colder than the model's domain: every sample takes the exact fits."""
    gp, prim, params = data
    cold = prim.clone()
    cold[1] *= 1e-4
    assert torch.equal(_trace(gp, cold, 33, coef=params), _trace(gp, cold, 33))


def test_no_plasma_at_all(data):
    gp, prim, params = data
    empty = prim.clone()
    empty[5:] = 0.0
    assert float(_trace(gp, empty, 33, coef=params).abs().max()) == 0.0

"""FP64 unpolarized images in two passes (samples, then the intensity): against the same image in
mixed precision (same geodesics, FP32 transfer) and against itself in waves, with and without
auxiliary images."""
import dataclasses
import math

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _trace(n, precision, aux, snaps=1, layout="planes", workspace=None, dtype=None,
           flags=native.BL_UNPOLARIZED):
    gp = S.grid_params_for(48, 32, 32)
    prim = torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()
    if snaps > 1:
        prim = torch.stack([prim.reshape(8, -1) * (1.0 + 0.1 * s) for s in range(snaps)]).contiguous()
        gp = dataclasses.replace(gp, n_snapshots=snaps, time_interp=1, t_first=0.0,
                                 dt_snapshots=40.0, t_camera=float(40 * snaps))
    if layout == "cells":
        prim, gp = images.pack_grid(prim, gp)
    dtype = dtype or (torch.float64 if precision == native.BL_PREC_FP64 else torch.float32)
    out = images.alloc_outputs(n, dtype, aux=aux)
    images.trace_images([S.Camera(theta=math.radians(60.0), n=n)],
                        [S.Metric(spin=0.9, precision=precision)], [gp], [prim], [230e9], outs=[out],
                        workspace=workspace, flags=flags)
    torch.cuda.synchronize()
    return torch.cat([out["stokes"].double()] + ([out["aux"].double()] if aux else []))


@pytest.mark.parametrize("n", [1, 33, 64])
@pytest.mark.parametrize("aux,snaps,layout", [(False, 1, "planes"), (True, 1, "cells"),
                                              (True, 3, "planes"), (False, 3, "cells")])
def test_against_mixed_and_in_waves(n, aux, snaps, layout):
    """FP32 transfer of the same geodesics: a few hundred additions of terms of one sign, each good
    to a few FP32 roundings, so 1e-4 of a plane's root mean square (without the emissivity-weighted
    means, whose weights underflow in FP32 at the image's faint edge); the waves and the FP32
    output bit for bit."""
    ref = _trace(n, native.BL_PREC_FP64, aux, snaps, layout)
    assert bool(torch.isfinite(ref).all()) and (n == 1 or float(ref[0].max()) > 0.0)
    got = _trace(n, native.BL_PREC_MIXED, aux, snaps, layout)
    rms = ref.flatten(1).square().mean(1).sqrt()
    err = (got - ref).flatten(1).square().mean(1).sqrt()
    weighted = torch.zeros_like(rms, dtype=torch.bool)
    weighted[4 + 12:4 + 19] = True
    assert bool(((err <= 1e-4 * rms) | weighted).all())
    small = torch.empty(6 << 20, dtype=torch.uint8, device="cuda")   # about 40 rays
    assert torch.equal(_trace(n, native.BL_PREC_FP64, aux, snaps, layout, small), ref)
    assert torch.equal(_trace(n, native.BL_PREC_FP64, aux, snaps, layout, dtype=torch.float32)[:4],
                       ref[:4].float().double())


@pytest.mark.parametrize("n", [1, 33])
def test_polarized_float32_output(n):
    """FP64 polarized images write the output's own type: rounded, and no plane beyond it."""
    ref = _trace(n, native.BL_PREC_FP64, False, flags=0)
    assert torch.equal(_trace(n, native.BL_PREC_FP64, False, dtype=torch.float32, flags=0),
                       ref.float().double())

"""The field mask of the grids and the FP32 sample pass against the paths they stand in for: a few
rays do not pay for a mask of the whole grid and run without one, and samples whose rows do not fit
beside the records run in the single-kernel transfer. Both change where a sample is looked up or
evaluated, not what is computed, so the same image must come out bit for bit."""
import dataclasses
import math

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu
FREQ = 230e9
# 16 chunks of 32 records a ray are stored; at this step limit the 32 x 32 image below fills 99 % of
# them and leaves room for 2800 sample rows, a tenth of what it needs
DS_MAX = 0.25


@pytest.fixture(scope="module", autouse=True)
def built():
    native.build()
    native.load()


def _patchy(nr, nt, nph, snaps=1):
    """A torus on a ragged grid, its field set to zero in seven of ten cells."""
    gp = S.grid_params_for(nr, nt, nph)
    prim = torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()
    prim = prim.reshape(8, nph, nt, nr)
    gen = torch.Generator().manual_seed(nr * 1000 + nt * 10 + nph)
    if snaps > 1:
        prim = torch.stack([prim * (1.0 + 0.1 * s) for s in range(snaps)])
        keep = (torch.rand((snaps, nph, nt, nr), generator=gen) > 0.7).float().cuda()
        prim[:, 5:] *= keep[:, None]
        gp = dataclasses.replace(gp, n_snapshots=snaps, time_interp=1, t_first=0.0,
                                 dt_snapshots=40.0, t_camera=float(40 * snaps))
    else:
        keep = (torch.rand((nph, nt, nr), generator=gen) > 0.7).float().cuda()
        prim[5:] *= keep
    return gp, prim.contiguous()


def _trace(jobs, precision, flags=0, coef=None, spin=0.9, incl=60.0):
    """jobs: (n, grid parameters, grid, metric options) an image; the first image's Stokes planes and
    records a ray."""
    cams = [S.Camera(theta=math.radians(incl), n=j[0]) for j in jobs]
    mets = [S.Metric(spin=spin, precision=precision, **j[3]) for j in jobs]
    dt = torch.float64 if precision == native.BL_PREC_FP64 else torch.float32
    outs = [images.alloc_outputs(j[0], dt, samples=True) for j in jobs]
    images.trace_images(cams, mets, [j[1] for j in jobs], [j[2] for j in jobs], [FREQ] * len(jobs),
                        outs=outs, flags=flags, coef_mlp=coef)
    torch.cuda.synchronize()
    return outs[0]["stokes"], outs[0]["samples"]


@pytest.mark.parametrize("precision", ["MIXED", "FAST"])
@pytest.mark.parametrize("dims,interp,layout,snaps", [
    ((65, 33, 40), 1, "cells", 1), ((65, 33, 40), 0, "planes", 1), ((600, 1, 40), 1, "planes", 1),
    ((600, 80, 1), 1, "cells", 1), ((65, 33, 40), 1, "cells", 3), ((33, 40, 31), 0, "cells", 2),
    ((1, 200, 200), 1, "cells", 1)])
def test_masked_and_unmasked_lookups_agree(precision, dims, interp, layout, snaps):
    """An 8 x 8 image is too few rays for its grid's mask alone (at most 256 cells a ray) and has
    one beside a 64 x 64 image of the same grid; plane-layout grids with learned coefficients."""
    gp, prim = _patchy(*dims, snaps)
    assert 256 * 64 < math.prod(dims) * snaps < 256 * 64 * 65
    coef = None
    if layout == "planes":
        coef = torch.empty(native.MLP_PARAMS, dtype=torch.float32, device="cuda")
        native.blacklight_mlp_init(coef, 5)
    gp = dataclasses.replace(gp, interp=interp)
    if layout == "cells":
        prim, gp = images.pack_grid(prim, gp)
    p = getattr(native, "BL_PREC_" + precision)
    alone = _trace([(8, gp, prim, {})], p, coef=coef)[0]
    assert torch.equal(_trace([(8, gp, prim, {}), (64, gp, prim, {})], p, coef=coef)[0], alone)


@pytest.mark.parametrize("precision", ["MIXED", "FAST"])
@pytest.mark.parametrize("unpolarized,snaps", [(False, 1), (True, 1), (False, 3), (True, 2)])
def test_rows_that_do_not_fit(precision, unpolarized, snaps):
    """Short steps through the whole grid fill the record store, so the samples' rows do not fit
    and the single kernel runs; in a batch with images that leave the store nearly empty they do."""
    gp = S.grid_params_for(48, 32, 32)
    prim = torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()
    if snaps > 1:
        prim = torch.stack([prim.reshape(8, -1) * (1.0 + 0.1 * s) for s in range(snaps)]).contiguous()
        gp = dataclasses.replace(gp, n_snapshots=snaps, time_interp=1, t_first=0.0,
                                 dt_snapshots=40.0, t_camera=float(40 * snaps))
    prim, gp = images.pack_grid(prim, gp)
    p = getattr(native, "BL_PREC_" + precision)
    flags = native.BL_UNPOLARIZED if unpolarized else 0
    dense = (32, gp, prim, dict(ds_max=DS_MAX))
    thin = (64, gp, prim, {})
    alone, records = _trace([dense], p, flags)
    assert int((records + 31).div(32, rounding_mode="floor").sum()) > 0.98 * 16 * 32 * 32
    assert float(alone[0].max()) > 0.0 and bool(torch.isfinite(alone).all())
    assert torch.equal(_trace([dense, thin], p, flags)[0], alone)

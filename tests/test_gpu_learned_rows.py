"""The learned form where the samples' rows do not fit beside the records (the single-kernel transfer
reads the model's outputs) against the same image in a batch whose other image leaves the store
nearly empty (they fit): the same bits, as for the exact fits in test_gpu_sample_pass."""
import dataclasses

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S
from test_gpu_sample_pass import DS_MAX, _trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["MIXED", "FAST"])
@pytest.mark.parametrize("snaps,cold", [(1, False), (3, False), (1, True)])
@pytest.mark.parametrize("incl", [60.0, 88.0])
def test_learned_rows_that_do_not_fit(precision, snaps, cold, incl):
    """cold: half of the grid below the model's temperature domain, so samples of both kinds."""
    native.build()
    native.load()
    gp = S.grid_params_for(48, 32, 32)
    prim = torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda()
    if cold:
        prim.view(8, 32, 32, 48)[1, :, :, 24:] *= 1e-4
    if snaps > 1:
        prim = torch.stack([prim.reshape(8, -1) * (1.0 + 0.1 * s) for s in range(snaps)]).contiguous()
        gp = dataclasses.replace(gp, n_snapshots=snaps, time_interp=1, t_first=0.0,
                                 dt_snapshots=40.0, t_camera=float(40 * snaps))
    prim, gp = images.pack_grid(prim, gp)
    model = torch.empty(native.MLP_PARAMS, dtype=torch.float32, device="cuda")
    native.blacklight_mlp_init(model, 5)
    p = getattr(native, "BL_PREC_" + precision)
    dense = (32, gp, prim, dict(ds_max=DS_MAX))
    thin = (64, gp, prim, {})
    alone, records = _trace([dense], p, coef=model, incl=incl)
    assert int((records + 31).div(32, rounding_mode="floor").sum()) > 0.98 * 16 * 32 * 32
    assert float(alone[0].max()) > 0.0 and bool(torch.isfinite(alone).all())
    both = _trace([dense, thin], p, coef=model, incl=incl)[0]
    bad = int((both != alone).sum())
    assert bad == 0, f"{bad} of {alone.numel()} values differ, by {float((both - alone).abs().max() / alone.abs().max()):.2e} of the largest"

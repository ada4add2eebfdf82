"""Field masks are built for the waves whose rays repay reading the grid, also where only the device
knows how many rays a wave has."""
import math

import pytest
import torch

from paper_2203_15963_gb300 import images, native
from paper_2203_15963_gb300 import synth as S

pytestmark = pytest.mark.gpu
FREQ = 230e9


@pytest.fixture(scope="module")
def grid():
    native.build()
    native.load()
    gp = S.grid_params_for(256, 128, 128)
    return images.pack_grid(torch.from_numpy(S.make_torus(gp, 0.9, S.BASE_SEED)).cuda(), gp)


def _mask_times(call):
    """Device time of each field_mask_kernel launch of call(), in us."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):   # (the first profile of a process may miss kernels)
        call()
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
    events = [e for e in prof.events() if "bl::" in e.name]
    if not events:
        pytest.skip("the profiler records no kernels here")
    return [e.device_time_total for e in events if "field_mask_kernel" in e.name]


def test_empty_levels_build_no_mask(grid):
    """A 64 x 64 root: 4.2e6 cells are too many for its 4096 rays, and a threshold that no block
    reaches leaves the finer levels without any, though they could hold 2.6e5. A 256 x 256 image of
    the same grid has its mask built."""
    cells, gp = grid
    cam = S.Camera(theta=math.radians(60.0), n=64)
    met = S.Metric(spin=0.9, precision=native.BL_PREC_FAST)
    out = {"stokes": torch.empty((4, 512, 512), dtype=torch.float32, device="cuda")}
    ad = native.adapt_struct(8, 3, native.BL_CRIT_ABS_GRAD, 1e300, 5)
    rays = []
    adaptive = _mask_times(lambda: rays.append(native.blacklight_trace_adaptive(
        [cam], [met], [gp], [cells], [FREQ], ad, [out])[1]))
    assert rays[-1].tolist() == [[64 * 64, 0, 0, 0]]
    big = images.alloc_outputs(256, torch.float32)
    built = _mask_times(lambda: images.trace_images(
        [S.Camera(theta=math.radians(60.0), n=256)], [met], [gp], [cells], [FREQ], outs=[big]))
    assert len(adaptive) == 4 and len(built) == 1
    assert max(adaptive) < 0.5 * built[0]
    # the composite is the root image, whose own trace has no mask either
    root = images.alloc_outputs(64, torch.float32)
    images.trace_images([cam], [met], [gp], [cells], [FREQ], outs=[root])
    assert torch.equal(out["stokes"][:, ::8, ::8], root["stokes"])

"""The program of the captures in this folder: two traces of one 256x256 image (a = 0.94, i = 60 deg)
of the 256x128x128 synthetic torus, cell layout, or a short training run.

    python profiles/one_image.py fp64|mixed|fast|learned|unpolarized|train [CTAs per SM]

A number of CTAs per SM traces through a plan with that configuration; for fp64 it selects the
64-warp kernels, which batches of more than 2560 rays an SM run.
"""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import torch

from paper_2203_15963_gb300 import coefmodel, images, native
from paper_2203_15963_gb300 import synth as S


def main(form, ctas=0):
    native.load()
    if form == "train":
        coefmodel.train(n=1 << 17, steps=20)
        torch.cuda.synchronize()
        return print("train: 2^17 samples, 20 steps of 16384")
    model = coefmodel.train(n=1 << 17, steps=200)[0] if form == "learned" else None
    fp64 = form in ("fp64", "unpolarized")
    cam, met, gp, prim = S.workload_inputs("torus256_cam256", 0.94, 60.0)
    met.precision = native.BL_PREC_FP64 if fp64 else \
        native.BL_PREC_MIXED if form == "mixed" else native.BL_PREC_FAST
    cells, gp = images.pack_grid(torch.from_numpy(prim).cuda(), gp)
    out = images.alloc_outputs(cam.n, torch.float64 if fp64 else torch.float32, samples=True)
    args = ([cam], [met], [gp], [cells], [230e9])
    if ctas:
        plan = native.Plan(*args, [out], config={"geo_ctas_per_sm": ctas, "tr_ctas_per_sm": ctas},
                           coef_mlp=model)
    for _ in range(2):
        if ctas:
            plan.run()
        else:
            images.trace_images(*args, outs=[out], coef_mlp=model,
                                flags=native.BL_UNPOLARIZED if form == "unpolarized" else 0)
    torch.cuda.synchronize()
    print(f"{form}: {int(out['steps'].sum())} attempts, {int(out['samples'].sum())} samples")


main(sys.argv[1], int(sys.argv[2]) if len(sys.argv) > 2 else 0)

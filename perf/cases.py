"""The work the ray tracer is used for, as measurable cases: images through every entry point a
program calls (single traces, batches on caller scratch, host buffers, captured plans, adaptive
plans) and the training of the learned coefficient model.

A case is a flat dict:
  kind       "trace" (blacklight_trace, library scratch), "batch" (trace_images with a caller
             workspace), "plan" (CUDA-graph replay), "adaptive" (adaptive plan), "host"
             (blacklight_trace_host_batch on pinned buffers) or "train" (coefmodel.train)
  precision  "fp64", "mixed" or "fast"
  n          pixels per side; spins, incs, freqs: comma-separated lists whose product is the
             batch (one fluid grid per spin, as in the repository's benchmark)
  nr, nt, nph, layout ("cells" / "planes"), interp (1 trilinear, 0 nearest), snapshots
  learned, unpolarized, aux: the coefficient model, Eq. unpolarized, the 26 auxiliary images
  integrator "dp", "rk4" or "rk2";  levels, block: adaptive refinement
  samples, steps, batch: training

Fluid data: the seeded synthetic torus of `synth` (density noise drawn on the device).
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2203_15963_gb300 import coefmodel, images, native
from paper_2203_15963_gb300 import synth as S

DEV = "cuda"
PRECISION = {"fp64": native.BL_PREC_FP64, "mixed": native.BL_PREC_MIXED,
             "fast": native.BL_PREC_FAST}
INTEGRATOR = {"dp": native.BL_INT_DP, "rk4": native.BL_INT_RK4, "rk2": native.BL_INT_RK2}
F_STEP = 0.02                  # RK4 / RK2 step factor
SNAP_DT, T_CAMERA = 10.0, 1035.0
EXACT_MAX_RAYS = 200_000       # a plain torch trace of more rays takes over about 20 s


def _image(kind, precision, n, spins, incs, grid, layout="cells", freqs="230e9", interp=1,
           snapshots=1, learned=False, unpolarized=False, aux=False, integrator="dp", levels=0,
           block=8):
    return dict(kind=kind, precision=precision, n=n, spins=spins, incs=incs, freqs=freqs,
                nr=grid[0], nt=grid[1], nph=grid[2], layout=layout, interp=interp,
                snapshots=snapshots, learned=learned, unpolarized=unpolarized, aux=aux,
                integrator=integrator, levels=levels, block=block)


SMALL, MEDIUM, LARGE = (64, 32, 32), (256, 128, 128), (512, 256, 256)


def listed():
    cases = [
        # one preview image of a small snapshot, as its file stores it: the smallest call, whose
        # time is the latency of the longest ray
        ("preview_fp64_32", _image("trace", "fp64", 32, "0.9", "17", SMALL, "planes")),
        # the plain FP64 method on a benchmark-sized snapshot, three spins in one batch
        ("batch_fp64_3x256", _image("batch", "fp64", 256, "0,0.5,0.94", "60", MEDIUM)),
        # FP64 geodesics with FP32 transfer at a camera size that no block size divides
        ("batch_mixed_2x201", _image("batch", "mixed", 201, "0.5,0.94", "17", MEDIUM)),
        # a parameter survey: nine images of three spins and three inclinations, fast form
        ("survey_fast_9x256", _image("batch", "fast", 256, "0,0.5,0.94", "17,60,90", MEDIUM)),
        # one odd-sized image of a snapshot left in the layout it arrives in
        ("planes_fast_301", _image("trace", "fast", 301, "0.94", "60", MEDIUM, "planes")),
        # the learned coefficient model at full resolution
        ("learned_fast_1024", _image("batch", "fast", 1024, "0.94", "17", LARGE, learned=True)),
        # slow light: eight snapshots, replayed as a plan (a frame of a movie)
        ("slowlight_plan_512", _image("plan", "fast", 512, "0.94", "60", MEDIUM, snapshots=8)),
        # adaptive refinement as a plan; FP64, whose refinement decisions do not hang on FP32
        # rounding
        ("adaptive_fp64_64", _image("adaptive", "fp64", 64, "0,0.94", "60", MEDIUM, levels=2)),
        # unpolarized image with the auxiliary images, FP64 (Eq. unpolarized, Sec. 4)
        ("aux_unpol_fp64_160", _image("batch", "fp64", 160, "0.94", "60", MEDIUM,
                                      unpolarized=True, aux=True)),
        # the fixed-rule RK4 integrator, FP32 transfer
        ("rk4_mixed_96", _image("batch", "mixed", 96, "0.5", "60", SMALL, integrator="rk4")),
        # end to end from host memory: grids copied in, images copied out
        ("host_fast_2x256", _image("host", "fast", 256, "0.5,0.94", "60", MEDIUM, "planes")),
        # training the learned model: data set, normalisation and the Adam steps
        ("train_model", dict(kind="train", samples=1 << 19, steps=4000, batch=16384)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "trace", "batch", "batch", "batch", "plan", "adaptive", "host",
                       "train"])
    if kind == "train":
        batch = 128 * _log_int(rng, 8, 128)
        return dict(kind="train", samples=_log_int(rng, 1 << 15, 1 << 19),
                    steps=_log_int(rng, 100, 4000), batch=batch)
    spin = lambda: "%.3f" % rng.uniform(0.0, 0.99)
    inc = lambda: "%.1f" % rng.uniform(5.0, 90.0)
    grid = (_log_int(rng, 48, 300), _log_int(rng, 24, 150), _log_int(rng, 24, 150))
    freqs = "%.4g" % rng.choice([86e9, 230e9, 345e9, 690e9])
    layout = rng.choice(["cells", "cells", "planes"])
    if kind == "adaptive":
        return _image(kind, "fp64", 8 * rng.randint(2, 8), spin(), inc(), grid, layout, freqs,
                      levels=rng.randint(1, 2), block=rng.choice([4, 8]))
    precision = rng.choice(["fp64", "mixed", "fast", "fast"])
    count = 1 if kind in ("trace", "plan") else rng.randint(1, 4)
    n = _log_int(rng, 17, 200 if precision == "fp64" else 400)
    if rng.random() < 0.3:
        n = max(16, n // 8 * 8)
    opts = {}
    if precision != "fp64" and kind in ("batch", "plan", "host") and rng.random() < 0.4:
        opts["learned"] = True
    elif kind == "batch" and rng.random() < 0.5:
        opts["unpolarized"] = rng.random() < 0.5
        opts["aux"] = rng.random() < 0.5
    if kind == "plan" and rng.random() < 0.5:
        opts["snapshots"] = rng.randint(2, 6)
    if kind == "batch" and not opts and rng.random() < 0.3:
        opts["integrator"] = rng.choice(["rk4", "rk2"])
        n = min(n, 100)
    if rng.random() < 0.2:
        opts["interp"] = 0
    return _image(kind, precision, n, ",".join(spin() for _ in range(count)), inc(), grid, layout,
                  freqs, **opts)


# ------------------------------------ inputs -----------------------------------------------
def _floats(text):
    return [float(v) for v in text.split(",")]


def _grid_params(case, layout="planes"):
    gp = S.GridParams(n_r=case["nr"], n_theta=case["nt"], n_phi=case["nph"],
                      interp=case["interp"],
                      layout=native.BL_GRID_CELLS if layout == "cells" else native.BL_GRID_PLANES)
    if case["snapshots"] > 1:
        gp = dataclasses.replace(gp, n_snapshots=case["snapshots"], dt_snapshots=SNAP_DT,
                                 t_camera=T_CAMERA)
    return gp


def _torus(case, gp, spin, seed):
    """The torus of synth.make_torus in the plane layout, its noise drawn on the device: the
    smooth part is axisymmetric, so one azimuth of it is made on the host."""
    flat = dataclasses.replace(gp, n_phi=1, n_snapshots=1)
    base = torch.from_numpy(S.make_torus(flat, spin, 0, noise=0.0)).to(DEV)
    gen = torch.Generator(DEV).manual_seed(seed)
    noise = torch.randn((gp.n_phi, gp.n_theta, gp.n_r), generator=gen, device=DEV)
    smooth = base.expand(8, gp.n_phi, gp.n_theta, gp.n_r)

    def snapshot(eps):
        p = smooth.clone()
        p[:2] *= (1.0 + 0.1 * eps).clamp(min=0.0)
        return p

    if gp.n_snapshots <= 1:
        return snapshot(noise)
    # the noise carried around by the Keplerian flow, in whole cells (synth.make_torus_series)
    omega = 1.0 / (torch.from_numpy(S.r_centres(gp)).to(DEV) ** 1.5 + spin)
    k = torch.arange(gp.n_phi, device=DEV)
    out = torch.empty((gp.n_snapshots,) + tuple(smooth.shape), device=DEV)
    for s in range(gp.n_snapshots):
        shift = torch.round(omega * s * gp.dt_snapshots / (2 * math.pi / gp.n_phi)).long()
        src = (k[:, None] - shift[None, :]) % gp.n_phi
        out[s] = snapshot(noise.gather(0, src[:, None, :].expand_as(noise)))
    return out


def _shape_targets(lx, lt):
    """The seven quantities the coefficient model learns, from the fits."""
    x = 10.0 ** lx
    u = x ** (-1.0 / 3.0)
    X = torch.sqrt(math.sqrt(2.0) * 1e3 / (1.5 * x))
    z = 10.0 ** (-lt)
    k0, k1 = torch.special.scaled_modified_bessel_k0(z), torch.special.scaled_modified_bessel_k1(z)
    k2 = k0 + 2.0 * k1 / z
    return torch.stack([
        torch.log(2.5651 * (1 + 1.92 * u + 0.9977 * u * u)),
        torch.log(2.5651 * (1 + 0.932 * u + 0.4998 * u * u)),
        torch.log(1.8138 / x + 3.423 * u * u + 0.02955 / torch.sqrt(x) + 2.0377 * u),
        2.011 * torch.exp(-X ** 1.035 / 4.7) - torch.cos(X / 2) * torch.exp(-X ** 1.2 / 2.73)
        - 0.011 * torch.exp(-X / 47.2),
        1.0 - 0.11 * torch.log1p(0.035 * X), torch.log(k2), torch.log(k0 / k2)], 1)


def _model(seed):
    """Weights of a coefficient model such as a program loads: random hidden layers, the output
    layer and the affine part by least squares on the fits."""
    gen = torch.Generator().manual_seed(seed)
    f = 2.0 * torch.rand((1 << 14, 3), generator=gen, dtype=torch.float64) - 1.0
    t = _shape_targets(1.5 + 4.5 * f[:, 0], 0.5 + 1.5 * f[:, 1])
    one = torch.ones((f.shape[0], 1), dtype=torch.float64)
    affine = torch.linalg.lstsq(torch.cat([f, one], 1), t).solution
    rest = t - torch.cat([f, one], 1) @ affine
    scale = rest.square().mean(0).sqrt()
    w1 = 2.0 * torch.randn((64, 4), generator=gen, dtype=torch.float64)
    w2 = torch.randn((64, 64), generator=gen, dtype=torch.float64) / 5.0
    b2 = 0.3 * torch.randn(64, generator=gen, dtype=torch.float64)
    w1, w2 = w1.bfloat16().double(), w2.bfloat16().double()
    h = torch.nn.functional.silu(torch.cat([f, one], 1) @ w1.T)
    h = torch.nn.functional.silu(h @ w2.T + b2)
    ridge = 1e-3 * torch.eye(65, dtype=torch.float64)
    hb = torch.cat([h, one], 1)
    w3 = torch.linalg.solve(hb.T @ hb + ridge, hb.T @ (rest / scale))
    p = torch.cat([w1.reshape(-1), w2.reshape(-1), b2, w3[:64].T.reshape(-1), w3[64], affine[3],
                   scale, affine[:3].T.reshape(-1)])
    return p.float().to(DEV)


def _setup(case, seed, layout):
    """Cameras, metrics, grid parameters, plane-layout grids (one per spin), frequencies."""
    cams, mets, gps, prims, freqs = [], [], [], [], []
    for k, spin in enumerate(_floats(case["spins"])):
        gp = _grid_params(case, layout)
        prim = _torus(case, gp, spin, 8 * seed + k)
        for inc in _floats(case["incs"]):
            for freq in _floats(case["freqs"]):
                cams.append(S.Camera(theta=math.radians(inc), n=case["n"]))
                mets.append(S.Metric(spin=spin, precision=PRECISION[case["precision"]],
                                     integrator=INTEGRATOR[case["integrator"]], f_step=F_STEP))
                gps.append(gp)
                prims.append(prim)
                freqs.append(freq)
    return cams, mets, gps, prims, freqs


def _pack(prims, gps):
    packed = {}
    for p, gp in zip(prims, gps):
        if id(p) not in packed:
            packed[id(p)] = images.pack_grid(p, dataclasses.replace(gp, layout=0))
    return [packed[id(p)][0] for p in prims], [packed[id(p)][1] for p in prims]


def prepare(case, seed):
    native.load()
    if case["kind"] == "train":
        return {"case": case, "seed": seed}
    cams, mets, gps, prims, freqs = _setup(case, seed, "planes")
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    model = _model(seed) if case["learned"] else None
    st = {"case": case, "model": model, "cams": cams, "mets": mets, "freqs": freqs,
          "flags": native.BL_UNPOLARIZED if case["unpolarized"] else 0}
    if case["kind"] == "host":
        hosts = {id(p): p.cpu().pin_memory() for p in prims}
        st["prims"], st["gps"] = [hosts[id(p)] for p in prims], gps
        st["model"] = None if model is None else model.cpu().pin_memory()
        st["outs"] = [{k: v.pin_memory() for k, v in
                       images.alloc_outputs(c.n, dt, device="cpu").items()} for c in cams]
        return st
    if case["layout"] == "cells":
        prims, gps = _pack(prims, gps)
    st["prims"], st["gps"] = prims, gps
    if case["kind"] == "adaptive":
        nf = case["n"] << case["levels"]
        st["outs"] = [{"stokes": torch.empty((4, nf, nf), dtype=dt, device=DEV)} for _ in cams]
        adapt = native.adapt_struct(case["block"], case["levels"], native.BL_CRIT_REL_GRAD, 0.1, 5)
        st["plan"] = native.AdaptivePlan(cams, mets, gps, prims, freqs, adapt, st["outs"])
        return st
    st["outs"] = [images.alloc_outputs(c.n, dt, device=DEV, aux=case["aux"]) for c in cams]
    if case["kind"] == "plan":
        st["plan"] = native.Plan(cams, mets, gps, prims, freqs, st["outs"], coef_mlp=model)
    elif case["kind"] == "batch":
        # the model's outputs take 32 bytes for each 64-byte record of the scratch
        need = native.blacklight_workspace_size(cams, mets)
        need = need * 3 // 2 if case["learned"] else need
        st["workspace"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        params, loss = coefmodel.train(seed=state["seed"], n=max(case["samples"], case["batch"]),
                                       batch=case["batch"], steps=case["steps"])
        return {"params": params, "loss": loss}
    args = (state["cams"], state["mets"], state["gps"], state["prims"], state["freqs"])
    if case["kind"] == "trace":
        native.blacklight_trace(*(a[0] for a in args), state["outs"][0])
    elif case["kind"] == "batch":
        images.trace_images(*args, outs=state["outs"], workspace=state["workspace"],
                            flags=state["flags"], coef_mlp=state["model"])
    elif case["kind"] == "host":
        native.blacklight_trace_host_batch(*args, state["outs"], coef_mlp=state["model"])
    else:
        state["plan"].run()
    return state["outs"]


def work(case):
    """One pass: the grids read and the outputs written once; per ray the adaptive integrator
    takes about 115 attempts of 1214 operations and 270 samples of 662 on these tori, a fixed-rule
    ray 2 ln(r_cam / r_hor) / f_step steps and as many samples."""
    if case["kind"] == "train":
        n = max(case["samples"], case["batch"])
        flops = 6.0 * 2 * (4 * 64 + 64 * 64 + 64 * 7) / 2 * case["batch"] * case["steps"]
        return {"bytes": 40.0 * n + 40.0 * case["batch"] * case["steps"] + 4.0 * 4906,
                "flops": flops + 1e3 * n}
    spins = len(_floats(case["spins"]))
    count = spins * len(_floats(case["incs"])) * len(_floats(case["freqs"]))
    pixels = count * case["n"] ** 2
    rays = pixels * (2.0 ** case["levels"] * 2.0 if case["levels"] else 1.0)
    grid = 32.0 * case["nr"] * case["nt"] * case["nph"] * case["snapshots"] * spins
    value = 8.0 if case["precision"] == "fp64" else 4.0
    planes = 4 + (26 if case["aux"] else 0)
    out = pixels * 4.0 ** case["levels"] * planes * value + (0 if case["levels"] else 8 * pixels)
    if case["integrator"] == "dp":
        per_ray = 115 * 1214 + 270 * (300 if case["unpolarized"] else 662)
    else:
        per_ray = 2 * math.log(500.0) / F_STEP * (4 * 130 + 662)
    if case["learned"]:
        per_ray += 27 * 2 * (4 * 64 + 64 * 64 + 64 * 7)
    return {"bytes": grid + out, "flops": rays * per_ray}


# --------------------------- the same images in plain 64-bit torch -----------------------------
# Every ray a column of float64 tensors. The method as the paper gives it: adaptive
# Dormand-Prince (or RK4 / RK2) geodesics in Cartesian Kerr-Schild coordinates, samples at step
# midpoints (or in equal parts of long steps), trilinear lookup, thermal synchrotron
# coefficients, transport of the coherency tensor, exact constant-coefficient Stokes steps.
DP_A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
        [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
        [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
        [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]
DP_B4 = [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40]
DP_MID = [6025192743 / 30085553152, 0, 51252292925 / 65400821598, -2691868925 / 45128329728,
          187940372067 / 1594534317056, -1776094331 / 19743644256, 11237099 / 235043384]


def _kerr(x, a):
    """r, f, l [3][n] and the derivatives d_c f [3][n], d_c l_b [3][3][n] at points x [3][n]."""
    R2 = (x * x).sum(0)
    q = R2 - a * a
    D = torch.sqrt(q * q + 4 * a * a * x[2] ** 2)
    r2 = 0.5 * (q + D)
    r = torch.sqrt(r2)
    s4, P = r2 * r2 + a * a * x[2] ** 2, r2 + a * a
    f = 2 * r * r2 / s4
    l = torch.stack([(r * x[0] + a * x[1]) / P, (r * x[1] - a * x[0]) / P, x[2] / r])
    dr = torch.stack([r * x[0] / D, r * x[1] / D, x[2] * P / (r * D)])
    ez = torch.zeros_like(x)
    ez[2] = 2 * a * a * x[2]
    df = f * (3 * dr / r - (4 * r2 * r * dr + ez) / s4)
    dl = torch.empty((3,) + tuple(x.shape), dtype=x.dtype, device=x.device)
    for c in range(3):
        dl[c, 0] = (dr[c] * x[0] + (r if c == 0 else 0) + (a if c == 1 else 0)
                    - 2 * r * dr[c] * l[0]) / P
        dl[c, 1] = (dr[c] * x[1] + (r if c == 1 else 0) - (a if c == 0 else 0)
                    - 2 * r * dr[c] * l[1]) / P
        dl[c, 2] = ((1 if c == 2 else 0) - l[2] * dr[c]) / r
    return r, f, l, df, dl


def _rhs(y, a):
    """dy/dl and r. The Kerr-Schild congruence has d_c l_b = A (delta_cb - l_c l_b) -
    B eps_cbk l_k with A + i B = 1 / (r - i a cos(theta)), and f = 2 A."""
    x, k = y[1:4], y[5:8]
    q, az2 = (x * x).sum(0) - a * a, (a * x[2]) ** 2
    D = torch.sqrt(q * q + 4 * az2)
    r2 = 0.5 * (q + D)
    r = torch.sqrt(r2)
    s4, P = r2 * r2 + az2, r2 + a * a
    A = r * r2 / s4
    f = 2 * A
    turned = torch.stack([a * x[1], -a * x[0], x[2] * (P / r - r)])
    l = (r * x + turned) / P
    lk = (l * k).sum(0)
    L = lk - y[4]
    dr = x * (r / D)
    dr[2] = dr[2] * (P / r2)
    df = (f * (3 / r - 4 * r2 * r / s4)) * dr
    df[2] -= 2 * a * a * x[2] * f / s4
    S = A * (k - lk * l) - (a * x[2] * r / s4) * torch.linalg.cross(k, l, dim=0)
    fL = f * L
    return torch.cat([(fL - y[4])[None], k - fL * l, torch.zeros_like(L)[None],
                      L * (0.5 * L * df + f * S)]), r


def _lower(f, l, v):
    ll = torch.cat([torch.ones_like(l[:1]), l])
    s = f * (ll * v).sum(0)
    out = v + s * ll
    out[0] = s - v[0]
    return out


def _raise(f, l, w):
    lu = torch.cat([-torch.ones_like(l[:1]), l])
    s = f * (lu * w).sum(0)
    out = w - s * lu
    out[0] = s - w[0]
    return out


def _camera(cam, a):
    """Camera position, K^a, H^a, V^a of a normal observer looking along k_i = (1, 0, 0)."""
    t = lambda v: torch.tensor(v, dtype=torch.float64)
    st, ct = math.sin(cam.theta), math.cos(cam.theta)
    x = t([st * cam.r, st * a, ct * cam.r]).reshape(3, 1)
    r, f, l, _, _ = _kerr(x, a)
    u = torch.cat([torch.sqrt(1 + f).reshape(1, 1), -f * l / torch.sqrt(1 + f)])
    ul = _lower(f, l, u)
    D = torch.sqrt(((x * x).sum(0) - a * a) ** 2 + 4 * a * a * x[2] ** 2)
    dr = torch.stack([r * x[0] / D, r * x[1] / D, x[2] * (r * r + a * a) / (r * D)])
    A, B = -1 - f, f * (l * dr).sum(0)
    C = (dr * dr).sum(0) - f * (l * dr).sum(0) ** 2
    k_t = (-B - torch.sqrt(B * B - A * C)) / A
    if not bool(A * k_t + B > 0):
        k_t = (-B + torch.sqrt(B * B - A * C)) / A
    kl = torch.cat([k_t.reshape(1, 1), dr])[:, 0]
    f, l, u, ul = f[0], l[:, 0], u[:, 0], ul[:, 0]
    ll = torch.cat([t([1.0]), l])
    g = torch.diag(t([-1.0, 1, 1, 1])) + f * torch.outer(ll, ll)
    gp = (g[1:, 1:] - torch.outer(ul[1:] / ul[0], g[0, 1:]) - torch.outer(g[1:, 0], ul[1:] / ul[0])
          + torch.outer(ul[1:], ul[1:]) / ul[0] ** 2 * g[0, 0])
    gi = torch.eye(3, dtype=torch.float64) - f * torch.outer(l, l) + torch.outer(u[1:], u[1:])
    Kl = kl[1:] - ul[1:] / ul[0] * kl[0]
    Kh, Kt = gi @ Kl, -(u * kl).sum()
    nk = 1 / torch.sqrt((Kl * Kh).sum())
    Kl, Kh, Kt = Kl * nk, Kh * nk, Kt * nk
    V = t([0.0, 0, 1]) - Kl[2] * Kh
    V = V / torch.sqrt(V @ gp @ V)
    H = torch.linalg.cross(gp @ V, Kl) / torch.sqrt(torch.det(gp))
    full = lambda w: torch.cat([(-(ul[1:] * w).sum() / ul[0]).reshape(1), w])
    return torch.cat([t([0.0]), x[:, 0]]), Kh + u[1:] * Kt, full(H), full(V)


def _rays(cams, mets):
    """Initial states y [8][rays], the spins, and H, V per ray, images after one another."""
    ys, spins, hs, vs = [], [], [], []
    for cam, met in zip(cams, mets):
        x, K, H, V = (v.to(DEV) for v in _camera(cam, met.spin))
        o = (torch.arange(cam.n, dtype=torch.float64, device=DEV) - 0.5 * cam.n + 0.5) \
            * cam.width / cam.n
        b, a = (v.reshape(-1) for v in torch.meshgrid(o, o, indexing="ij"))
        pos = x[:, None] + a * H[:, None] + b * V[:, None]
        spin = torch.full_like(a, met.spin)
        _, f, l, _, _ = _kerr(pos[1:], spin)
        lk = (l * K[:, None]).sum(0)
        A, B, C = f - 1, f * lk, (K * K).sum() + f * lk * lk
        k = torch.cat([((-B - torch.sqrt(B * B - A * C)) / A)[None], K[:, None].expand(3, a.numel())])
        ys.append(torch.cat([pos, _lower(f, l, k)]))
        spins.append(spin)
        hs.append(H[:, None].expand(4, a.numel()))
        vs.append(V[:, None].expand(4, a.numel()))
    return torch.cat(ys, 1), torch.cat(spins), torch.cat(hs, 1), torch.cat(vs, 1)


class _Records:
    """Samples of all rays [records][14][rays]: sample x, k; node x, k; length; time."""

    def __init__(self, rays):
        self.n = torch.zeros(rays, dtype=torch.long, device=DEV)
        self.v = torch.zeros((128, 14, rays), dtype=torch.float64, device=DEV)

    def add(self, rays, sample, node, dl):
        at = self.n[rays]
        if at.numel() and int(at.max()) >= self.v.shape[0]:
            self.v = torch.cat([self.v, torch.zeros_like(self.v)])
        v = torch.cat([sample[1:4], sample[5:8], node[1:4], node[5:8], dl[None], sample[:1]])
        self.v[at, :, rays] = v.T
        self.n[rays] += 1

    def get(self, i):
        return self.v[i]


def _emit(rec, rays, met, r_max, h, rates, rs, mid, interior, y0):
    """Records of accepted steps: one at the midpoint, or ds / ds_max equal parts."""
    r, f, l, _, _ = _kerr(mid[1:4], rates["a"])
    L = (l * mid[5:8]).sum(0) - mid[4]
    ds = h.abs() * (f * L - mid[4]).abs() / torch.sqrt(1 + f)
    near = torch.minimum(r, torch.minimum(*rs)) < r_max
    parts = torch.where(near & (ds > met.ds_max), torch.ceil(ds / met.ds_max), torch.ones_like(ds))
    for s in range(int(parts.max())):
        m = parts > s
        whole, p = (parts == 1)[m], parts[m]
        smp = torch.where(whole, mid[:, m], interior((s + 0.5) / p, m))
        node = y0[:, m] if s == 0 else interior(s / p, m)
        rec.add(rays[m], smp, node, h[m].abs() / p)
    return ds


def _geodesics(cams, mets, r_max):
    met = mets[0]
    y, spin, H, V = _rays(cams, mets)
    n = y.shape[1]
    r_hor = 1 + torch.sqrt(1 - spin * spin)
    r_cam, r_in = cams[0].r, met.r_in_over_rhor * r_hor
    rec = _Records(n)
    end_t, length, affine = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(3))
    live = torch.arange(n, device=DEV)
    k0, r = _rhs(y, spin)
    inside = r < r_cam
    kt, a = y[4].clone(), spin
    h = -met.h0_frac * (r_cam - r_hor)
    rejected = torch.zeros(n, dtype=torch.bool, device=DEV)
    while live.numel():
        if met.integrator == native.BL_INT_DP:
            k = [k0]
            for row in DP_A[1:]:
                ys = y + h * sum(w * q for w, q in zip(row, k) if w != 0)
                d, r1 = _rhs(ys, a)
                k.append(d)
            y1, k1 = ys, k[6]
            err = (h * sum((b - e) * q for b, e, q in zip(DP_A[6] + [0.0], DP_B4, k))).abs()
            eps = (err / (met.tol_abs + met.tol_rel * torch.maximum(y.abs(), y1.abs()))).amax(0)
            ok = eps <= 1
            fac = torch.where(eps == 0, torch.full_like(eps, 10.0), 0.9 * eps ** -0.2).clamp(0.2, 10)
            fac = torch.where(ok & ~rejected, fac, fac.clamp(max=1.0))
            mid = y + 0.5 * h * sum(w * q for w, q in zip(DP_MID, k) if w != 0)
        else:
            h = -met.f_step * (r - (1 + torch.sqrt(1 - a * a)))
            if met.integrator == native.BL_INT_RK4:
                q2 = _rhs(y + 0.5 * h * k0, a)[0]
                q3 = _rhs(y + 0.5 * h * q2, a)[0]
                q4 = _rhs(y + h * q3, a)[0]
                y1 = y + h * (k0 / 6 + q2 / 3 + q3 / 3 + q4 / 6)
            else:
                y1 = y + h * 0.5 * (k0 + _rhs(y + h * k0, a)[0])
            k1, r1 = _rhs(y1, a)
            ok = torch.ones_like(r1, dtype=torch.bool)
            fac = torch.ones_like(r1)
            mid = 0.5 * (y + y1) + 0.125 * h * (k0 - k1)
        d0 = h * k0
        D1, D2, D3 = y1 - y - d0, h * k1 - d0, mid - y - 0.5 * d0
        quart = (-5 * D1 + D2 + 16 * D3, 14 * D1 - 3 * D2 - 32 * D3, -8 * D1 + 2 * D2 + 16 * D3)
        w = ok.nonzero()[:, 0]

        def interior(t, m):
            c = w[m]
            q = [v[:, c] for v in quart]
            return y[:, c] + t * (d0[:, c] + t * (q[0] + t * (q[1] + t * q[2])))

        if w.numel():
            ds = _emit(rec, live[w], met, r_max, h[w], {"a": a[w]}, (r[w], r1[w]), mid[:, w],
                       interior, y[:, w])
            length[live[w]] += ds
            affine[live[w]] += h[w].abs()
        y, k0 = torch.where(ok, y1, y), torch.where(ok, k1, k0)
        r = torch.where(ok, r1, r)
        h, rejected = h * fac, ~ok
        done = ok & ((r < 1.01 * (1 + torch.sqrt(1 - a * a))) | (inside & (r > r_cam)))
        inside = inside | (r < r_cam)
        end_t[live[done]] = y[0][done]
        keep = ~done
        live, y, k0, r, h, a = live[keep], y[:, keep], k0[:, keep], r[keep], h[keep], a[keep]
        inside, rejected = inside[keep], rejected[keep]
    return rec, kt, spin, H, V, (-end_t, length, affine)


def _lookup(gp, grids, which, x, t, r, a):
    """Primitives [8][n] at points, grids [G][snapshots][8][nph][nt][nr] flattened."""
    cth = (x[2] / r).clamp(-1, 1)
    ph = torch.atan2(x[1] * r - x[0] * a, x[0] * r + x[1] * a) % (2 * math.pi)
    u = [torch.log(r / gp.r_min) / (math.log(gp.r_max / gp.r_min) / gp.n_r),
         torch.acos(cth) * gp.n_theta / math.pi, ph * gp.n_phi / (2 * math.pi)]
    dims = (gp.n_r, gp.n_theta, gp.n_phi)

    def cells(at):                              # ([lower, upper], weight of upper) per axis
        if not gp.interp:
            lo = [torch.floor(v).long().clamp(0, d - 1) for v, d in zip(at, dims)]
            return [(i, i, torch.zeros_like(r)) for i in lo]
        out = []
        for c, (v, d) in enumerate(zip(at, dims)):
            v = v - 0.5
            if c < 2:
                v = v.clamp(0, d - 1)
                i = torch.floor(v).long().clamp(max=max(d - 2, 0))
                out.append((i, (i + 1).clamp(max=d - 1), v - i))
            else:
                i = torch.floor(v).long()
                out.append((i % d, (i + 1) % d, v - i))
        return out

    (i0, i1, wi), (j0, j1, wj), (k0, k1, wk) = cells(u)
    plane = gp.n_r * gp.n_theta * gp.n_phi
    v8 = torch.arange(8, device=DEV)[:, None] * plane

    def snapshot(s):
        base = (which * max(1, gp.n_snapshots) + s) * 8 * plane
        out = 0
        for k, wk_ in ((k0, 1 - wk), (k1, wk)):
            for j, wj_ in ((j0, 1 - wj), (j1, wj)):
                for i, wi_ in ((i0, 1 - wi), (i1, wi)):
                    out = out + wk_ * wj_ * wi_ * grids[v8 + base + (k * gp.n_theta + j) * gp.n_r + i]
        return out, cth, ph

    if gp.n_snapshots <= 1:
        return snapshot(0)
    ts = ((t + gp.t_camera - gp.t_first) / gp.dt_snapshots).clamp(0, gp.n_snapshots - 1)
    s0 = torch.floor(ts).long().clamp(max=gp.n_snapshots - 2)
    w = ts - s0
    return (1 - w) * snapshot(s0)[0] + w * snapshot(s0 + 1)[0], cth, ph


def _plasma(gp, grids, which, x, t, a, geom):
    """u^a, b^a and the plasma quantities of samples inside the grid, and which carry plasma."""
    r, f, l = geom
    p, cth, ph = _lookup(gp, grids, which, x, t, r, a)
    sth = torch.sqrt(1 - cth * cth)
    az = torch.hypot(x[0] * r + x[1] * a, x[1] * r - x[0] * a) > 0
    cp, sp = torch.where(az, torch.cos(ph), 0.0), torch.where(az, torch.sin(ph), 0.0)
    J = ((sth * cp, cth * (r * cp - a * sp), sth * (-r * sp - a * cp)),
         (sth * sp, cth * (r * sp + a * cp), sth * (r * cp - a * sp)), (cth, -r * sth, 0 * r))
    v = torch.stack([sum(J[c][k] * p[2 + k] for k in range(3)) for c in range(3)])
    B = torch.stack([sum(J[c][k] * p[5 + k] for k in range(3)) for c in range(3)])
    un = torch.sqrt(1 + (v * v).sum(0) + f * (l * v).sum(0) ** 2)
    ut = un * torch.sqrt(1 + f)
    u = torch.cat([ut[None], v - f / (1 + f) * ut * l])
    ul = _lower(f, l, u)
    bt = (B * ul[1:]).sum(0)
    b = torch.cat([bt[None], (B + bt * u[1:]) / ut])
    bsq = (b * _lower(f, l, b)).sum(0)
    rho, pg = p[0], (gp.gamma_ad - 1) * p[1]
    ok = torch.isfinite(p).all(0) & (rho > 0) & (pg > 0) & (bsq > 0) & ~(bsq / rho > gp.sigma_cut)
    binv = bsq / (2 * pg)
    ratio = (gp.r_high + binv ** 2 * gp.r_low) / (1 + binv ** 2)
    th = gp.mu * M_P / M_E * pg / rho * (gp.ne_over_ni + 1) / (gp.ne_over_ni + ratio)
    ne = rho * gp.rho_unit_cgs / (gp.mu * M_P) / (1 + 1 / gp.ne_over_ni)
    bg = torch.sqrt(bsq) * C_CGS * math.sqrt(4 * math.pi * gp.rho_unit_cgs)
    return u, ul, b, bsq, rho, ne, pg, th, bg, binv, ok


C_CGS, E_CGS, M_E, M_P = 2.99792458e10, 4.80320471e-10, 9.1093837015e-28, 1.67262192369e-24
H_CGS, G_CGS, M_SUN = 6.62607015e-27, 6.67430e-8, 1.98841e33


def _coefficients(ne, th, bg, nu, cth):
    """j_I, j_Q, j_V, alpha_I, alpha_Q, alpha_V, rho_Q, rho_V of thermal electrons."""
    sth = torch.sqrt((1 - cth * cth).clamp(min=0))
    nub = E_CGS * bg / (2 * math.pi * M_E * C_CGS)
    z = 1 / th
    k0, k1 = torch.special.scaled_modified_bessel_k0(z), torch.special.scaled_modified_bessel_k1(z)
    k2 = k0 + 2 * th * k1
    x = nu / (1.5 * nub * sth * th * th)
    x13 = x ** (1 / 3)
    ex = torch.exp(z - 1.8899 * x13) / k2
    pre = ne * E_CGS ** 2 / (math.sqrt(3) * C_CGS) * nu
    j = [pre * 2.5651 * (1 + 1.92 / x13 + 0.9977 / x13 ** 2) * ex,
         pre * 2.5651 * (1 + 0.932 / x13 + 0.4998 / x13 ** 2) * ex,
         pre * 4 / 3 * z * cth / sth * ex * (1.8138 / x + 3.423 / x13 ** 2 + 0.02955 / torch.sqrt(x)
                                             + 2.0377 / x13)]
    ib = torch.expm1(H_CGS * nu / (M_E * C_CGS ** 2) * z) * (C_CGS / nu) ** 2 / (2 * H_CGS * nu)
    X = th * torch.sqrt(math.sqrt(2) * 1e3 * sth * nub / nu)
    fm = 2.011 * torch.exp(-X ** 1.035 / 4.7) - torch.cos(X / 2) * torch.exp(-X ** 1.2 / 2.73) \
        - 0.011 * torch.exp(-X / 47.2)
    base = ne * E_CGS ** 2 / (M_E * C_CGS)
    rq = base * (nub * sth) ** 2 / nu ** 3 * fm * (k1 / k2 + 6 * th)
    rv = 2 * base * nub * cth / nu ** 2 * k0 / k2 * (1 - 0.11 * torch.log1p(0.035 * X))
    return j + [v * ib for v in j] + [rq, rv]


def _frame(f, l, u, ul, b, kl):
    """e1, e2 of the fluid frame: e3 along the photon, e2 along the projected field."""
    ku = _raise(f, l, kl)
    w = -(kl * u).sum(0)
    e3, e3l = ku / w - u, kl / w - ul
    bp = b + (b * ul).sum(0) * u
    bp = bp - (bp * e3l).sum(0) * e3
    e2 = bp / torch.sqrt((bp * _lower(f, l, bp)).sum(0))
    e2l = _lower(f, l, e2)
    # e1^a = [abcd] u_b e2_c e3_d
    cross = lambda p, q: torch.linalg.cross(p[1:], q[1:], dim=0)
    n = cross(e2l, e3l)
    e1 = torch.cat([(ul[1:] * n).sum(0)[None],
                    -ul[0] * n + e2l[0] * cross(ul, e3l) - e3l[0] * cross(ul, e2l)])
    return e1, e2


def _expm(Z):
    """exp of [n][5][5]: Taylor polynomial of Z / 2^s, squared s times."""
    s = max(0, int(torch.ceil(torch.log2(Z.abs().sum(2).max().clamp(min=1e-3) / 0.5))))
    Z = Z / 2.0 ** s
    one = torch.eye(5, dtype=Z.dtype, device=Z.device)
    E = one + Z / 15
    for k in range(14, 0, -1):
        E = one + Z @ E / k
    for _ in range(s):
        E = E @ E
    return E


def _transport(x, kl, a):
    """A^a_d = -k^c Gamma^a_cd, [4][4][n]."""
    r, f, l, df, dl = _kerr(x, a)
    k = _raise(f, l, kl)
    n = x.shape[1]
    ll = torch.cat([torch.ones_like(l[:1]), l])
    dg = torch.zeros((4, 4, 4, n), dtype=x.dtype, device=x.device)
    dl4 = torch.zeros((4, 4, n), dtype=x.dtype, device=x.device)
    dl4[1:, 1:] = dl
    df4 = torch.cat([torch.zeros_like(df[:1]), df])
    dg = df4[:, None, None] * ll[:, None] * ll + f * (dl4[:, :, None] * ll + ll[:, None] * dl4[:, None])
    D = (k[:, None, None] * dg).sum(0)                     # k^c d_c g_ed
    P = (dg * k[None, :, None]).sum(1)                     # P[m][e] = d_m g_ec k^c
    C = 0.5 * (D + P.transpose(0, 1) - P)                  # C_ed = k^c Gamma_ecd
    lu = torch.cat([-torch.ones_like(l[:1]), l])
    raised = C.clone()
    raised[0] = -C[0]
    return f * lu[:, None] * (lu[:, None] * C).sum(0) - raised


def _image64(case, seed):
    cams, mets, gps, prims, freqs = _setup(case, seed, "planes")
    gp, n = gps[0], case["n"] ** 2
    order = list(dict.fromkeys(id(p) for p in prims))
    grids = torch.cat([next(p for p in prims if id(p) == i).reshape(-1) for i in order]).double()
    per = lambda vals, dt=torch.float64: torch.tensor(vals, dtype=dt, device=DEV).repeat_interleave(n)
    which, freq = per([order.index(id(p)) for p in prims], torch.long), per(freqs)
    rec, kt, spin, H, V, path = _geodesics(cams, mets, gp.r_max)
    rays = kt.numel()
    unit = G_CGS * gp.mass_msun * M_SUN / C_CGS ** 2
    N = torch.zeros((4, 4, rays), dtype=torch.complex128, device=DEV)
    intensity = torch.zeros(rays, dtype=torch.float64, device=DEV)
    lit = torch.zeros(rays, dtype=torch.bool, device=DEV)
    Ij, tau = torch.zeros_like(intensity), torch.zeros_like(intensity)
    Q = torch.zeros((3, 7, rays), dtype=torch.float64, device=DEV)

    def step(m, at, h):
        """Predictor-corrector of the coherency tensor from record `at` on, rays m."""
        v = rec.get(at)[:, m]
        A0 = _transport(v[:3], torch.cat([kt[m][None], v[3:6]]), spin[m])
        A1 = _transport(v[6:9], torch.cat([kt[m][None], v[9:12]]), spin[m])
        cur = N[:, :, m]
        F = lambda A, T: (lambda AT: AT + AT.transpose(0, 1).conj())((A[:, :, None] * T[None]).sum(1))
        half = cur + 0.5 * h * F(A0, cur)
        N[:, :, m] = cur + h * F(A1, half)

    for i in range(int(rec.n.max()) - 1, -1, -1):
        here = rec.n > i
        if not case["unpolarized"]:
            m = (here & lit).nonzero()[:, 0]
            if m.numel():
                step(m, i + 1, 0.5 * (rec.get(i + 1)[12, m] + rec.get(i)[12, m]))
        v = rec.get(i)
        r = _kerr(v[:3], spin)[0] if here.all() else torch.where(
            here, _kerr(torch.where(here, v[:3], 100.0), spin)[0], 1e9)
        m = (here & (r >= gp.r_min) & (r <= gp.r_max)).nonzero()[:, 0]
        if not m.numel():
            continue
        r, f, l, _, _ = _kerr(v[:3, m], spin[m])
        state = _plasma(gp, grids, which[m], v[:3, m], v[13, m], spin[m], (r, f, l))
        ok = state[-1]
        if not bool(ok.any()):
            continue
        m, f, l = m[ok], f[ok], l[:, ok]
        u, ul, b, bsq, rho, ne, pg, th, bg, binv = (s[..., ok] for s in state[:-1])
        kl, dl = torch.cat([kt[m][None], v[3:6, m]]), v[12, m]
        w, kb = -(kl * u).sum(0), (kl * b).sum(0)
        nu = freq[m] / -kt[m] * w
        co = _coefficients(ne, th, bg, nu, (kb / (w * torch.sqrt(bsq))).clamp(-1, 1))
        path_l = unit * w
        e = [c * (freq[m] / nu) ** 3 * path_l for c in co[:3]]
        al = [c * path_l for c in co[3:]]
        if case["aux"]:
            q = torch.stack([rho, ne, pg, th, bg, bsq / rho, binv])
            dt = al[0] * dl
            Ij[m] += e[0] * dl
            tau[m] += dt
            Q[0][:, m] += q * dl
            Q[1][:, m] += q * e[0] * dl
            Q[2][:, m] = torch.exp(-dt) * Q[2][:, m] - torch.expm1(-dt) * q
        if case["unpolarized"]:
            dt = al[0] * dl
            thin = intensity[m] * torch.exp(-dt) - torch.expm1(-dt) * e[0] / al[0]
            intensity[m] = torch.where(al[0] > 0, torch.where(dt >= 100, e[0] / al[0], thin),
                                       intensity[m] + e[0] * dl)
            continue
        e1, e2 = _frame(f, l, u, ul, b, kl)
        e1l, e2l = _lower(f, l, e1), _lower(f, l, e2)
        con = lambda p, q: (p[:, None] * q[None] * N[:, :, m]).sum((0, 1))
        n11, n22, n12 = con(e1l, e1l).real, con(e2l, e2l).real, con(e1l, e2l)
        s = torch.stack([n11 + n22, n11 - n22, 2 * n12.real, 2 * n12.imag], 1)
        z = torch.zeros_like(dl)
        M = torch.stack([torch.stack(row, 1) for row in
                         ((al[0], al[1], z, al[2]), (al[1], al[0], al[4], z),
                          (z, -al[4], al[0], al[3]), (al[2], z, -al[3], al[0]))], 1)
        Jv = torch.stack([e[0], e[1], z, e[2]], 1)
        big = torch.zeros((m.numel(), 5, 5), dtype=torch.float64, device=DEV)
        thick = al[0] * dl >= 100
        big[:, :4, :4] = torch.where(thick[:, None, None], 0.0, -M * dl[:, None, None])
        big[:, :4, 4] = Jv * dl[:, None]
        E = _expm(big)
        s1 = (E[:, :4, :4] @ s[:, :, None])[:, :, 0] + E[:, :4, 4]
        if bool(thick.any()):
            s1[thick] = torch.linalg.solve(M[thick], Jv[thick])
        p, q_, uu, vv = 0.5 * (s1[:, 0] + s1[:, 1]), 0.5 * (s1[:, 0] - s1[:, 1]), s1[:, 2] / 2, s1[:, 3] / 2
        o11, o22, o12 = e1[:, None] * e1, e2[:, None] * e2, e1[:, None] * e2
        N[:, :, m] = p * o11 + q_ * o22 + torch.complex(uu, vv) * o12 \
            + torch.complex(uu, -vv) * o12.transpose(0, 1)
        lit[m] = True
    if case["unpolarized"]:
        stokes = torch.stack([intensity] + [torch.zeros_like(intensity)] * 3)
    else:
        m = lit.nonzero()[:, 0]
        if m.numel():
            step(m, 0, 0.5 * rec.get(0)[12, m])
        r, f, l, _, _ = _kerr(rec.get(0)[6:9], spin)
        hl, vl = _lower(f, l, H), _lower(f, l, V)
        con = lambda p, q: (p[:, None] * q[None] * N).sum((0, 1))
        n11, n22, n12 = con(hl, hl).real, con(vl, vl).real, con(hl, vl)
        stokes = torch.stack([n11 + n22, n11 - n22, 2 * n12.real, 2 * n12.imag])
    aux = None
    if case["aux"]:
        mean = torch.where(Ij > 0, Q[1] / Ij, 0.0)
        aux = torch.cat([torch.stack(path + (Ij, tau)), Q[0] / path[2], mean, Q[2]])
    out = []
    for k, cam in enumerate(cams):
        cut = slice(k * n, (k + 1) * n)
        o = {"stokes": stokes[:, cut].reshape(4, cam.n, cam.n), "status": None, "steps": None}
        if case["aux"]:
            o["aux"] = aux[:, cut].reshape(26, cam.n, cam.n)
        out.append(o)
    return out


def exact(case, seed):
    """The images in 64 bits; None for the learned model (bf16 weights and activations are its
    definition, in training and in use), for adaptive composites (their blocks follow from
    thresholds) and where the plain trace takes too long."""
    if case["kind"] in ("train", "adaptive") or case["learned"]:
        return None
    rays = case["n"] ** 2 * len(_floats(case["spins"])) * len(_floats(case["incs"]))
    if rays > EXACT_MAX_RAYS:
        return None
    return _image64(case, seed)

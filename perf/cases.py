"""Performance cases: the work that users of this package have it do, through its
public entry points, as single passes that can be timed and compared.

Two families, in the proportions of the package's own workloads:

* Monte Carlo photon runs (``spmc``): Cahn-Hilliard pore masks from small odd
  crops up to 512^3, the voxel-field and the depth-profile tally, FP32 and FP64
  transport, periodic and mirror lateral faces, single runs and batched launches.
  A pass returns the integer tallies, the FP64 estimators and the voxel field.
* The fluence surrogate (``spnn``): single layers (forward, input gradient, weight
  and bias gradient), inference from mask to profiles, and a gradient step of the
  whole U-Net.

``listed()`` are the named cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes what a program has in hand before the call, ``run`` is one pass,
``work`` the bytes and operations the pass cannot do without, ``exact`` the same
outputs in 64 bits where plain arithmetic gives them in seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_13929_gb300 import inputs, spmc, spnn

MUS, MUA, G = 0.5, 0.005, 0.7          # the benchmark optics of the solid, per voxel
KINDS = {"conv3": spnn.CONV3, "down": spnn.DOWN, "up": spnn.UP}
TAPS = {"conv3": 27, "down": 8, "up": 8}


# ------------------------------------------------------------------- cases --

def listed():
    mc = {"kind": "mc", "tally": "field", "precision": 32, "mirror": 0, "mu_s": MUS, "mu_a": MUA, "g": G}
    return [
        # One whole simulation of a small mask that is already on the GPU, few photons, no
        # allocation: the latency of a call inside a host application's loop.
        {"name": "mc_noalloc_64", "kind": "noalloc", "nx": 64, "ny": 64, "nz": 64, "phi": 0.70,
         "mu_s": MUS, "mu_a": MUA, "g": G, "photons": 20_000},
        # The plain 64^3 phi = 0.70 configuration at its 2e5 photons with the voxel fluence:
        # the ordinary small run.
        dict(mc, name="mc_64_field", nx=64, ny=64, nz=64, phi=0.70, photons=200_000),
        # The paper-scale 256^3 phi = 0.90 mask with the full voxel field (the headline workload,
        # fewer photons per pass).
        dict(mc, name="mc_256_field", nx=256, ny=256, nz=256, phi=0.90, photons=5_000_000),
        # The paper-scale phi = 0.70 mask when only depth profiles and R/T/A are wanted.
        dict(mc, name="mc_256_profile", nx=256, ny=256, nz=256, phi=0.70, tally="profile", photons=5_000_000),
        # The precision study's 512^3 mask: a 1 GiB voxel field, far larger than L2.
        dict(mc, name="mc_512_field", nx=512, ny=512, nz=512, phi=0.90, photons=2_000_000),
        # FP64 transport (the precision study's other arm) on a small odd-sized mask with the
        # paper's mirror faces.
        dict(mc, name="mc_fp64_odd", nx=75, ny=50, nz=99, phi=0.90, precision=64, mirror=1, photons=50_000),
        # The surrogate's data pipeline: 16 masks of 64^3 in one batched run, then the
        # log-fluence training targets.
        {"name": "batch_targets_64", "kind": "batch", "count": 16, "sizes": "64", "photons": 1_000_000,
         "targets": True},
        # A design sweep over masks of uneven size and optics in one persistent launch, run
        # after run on the same handle.
        {"name": "batch_uneven", "kind": "batch", "count": 8, "sizes": "64,96,128,160,192,224,256",
         "photons": 500_000, "targets": False},
        # One training pass of the U-Net's commonest layer: conv3 32 -> 32 on 64^3.
        {"name": "conv3_64", "kind": "layer", "layer": "conv3", "B": 16, "D": 64, "H": 64, "W": 64,
         "c0": 32, "c1": 0, "cout": 32},
        # The same for a decoder layer that reads [up, skip] at half resolution.
        {"name": "conv3_32_concat", "kind": "layer", "layer": "conv3", "B": 16, "D": 32, "H": 32, "W": 32,
         "c0": 64, "c1": 64, "cout": 64},
        # Screening one mask: features, network, depth profiles, batch of one.
        {"name": "unet_predict_1", "kind": "predict", "c0": 32, "n": 64, "batch": 1},
        # A gradient step of the whole network at a training batch.
        {"name": "unet_grad_64", "kind": "grad", "c0": 32, "n": 64, "batch": 64},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _optics(rng):
    """Optics of the batched configuration, or the benchmark's own."""
    if rng.random() < 0.4:
        return {"mu_s": MUS, "mu_a": MUA, "g": G}
    return {"mu_s": round(_log_uniform(rng, 0.1, 2.0), 4), "mu_a": round(rng.uniform(0.001, 0.05), 4),
            "g": round(rng.uniform(0.0, 0.9), 3)}


def _photons(rng, case, lo, hi):
    """Photon count whose voxel steps are log-uniform in [lo, hi], at most 5e6 photons."""
    return max(1000, min(5_000_000, int(_log_uniform(rng, lo, hi) / _steps_per_photon(case))))


def draw(rng):
    kind = rng.choices(["mc", "noalloc", "batch", "layer", "predict", "grad"], [7, 2, 3, 5, 2, 2])[0]
    if kind == "noalloc":
        c = {"kind": kind, "nx": int(_log_uniform(rng, 20, 160)), "ny": int(_log_uniform(rng, 20, 160)),
             "nz": int(_log_uniform(rng, 16, 160)), "phi": round(rng.uniform(0.5, 0.95), 3), **_optics(rng)}
        c["photons"] = _photons(rng, c, 1e6, 2e8)
        return c
    if kind == "mc":
        p = rng.random()
        c = {"kind": kind, "tally": "field" if rng.random() < 0.7 else "profile",
             "precision": 64 if p < 0.12 else 32, "mirror": 1 if rng.random() < 0.25 else 0}
        hi = 128 if c["precision"] == 64 else 320
        c.update(nx=int(_log_uniform(rng, 24, hi)), ny=int(_log_uniform(rng, 24, hi)),
                 nz=int(_log_uniform(rng, 16, hi)), phi=round(rng.uniform(0.5, 0.95), 3), **_optics(rng))
        c["photons"] = _photons(rng, c, 1e6, 3e7) if c["precision"] == 64 else _photons(rng, c, 1e7, 3e9)
        return c
    if kind == "batch":
        if rng.random() < 0.5:
            return {"kind": kind, "count": rng.randint(4, 24), "sizes": str(rng.choice([48, 64, 72])),
                    "photons": int(_log_uniform(rng, 1e5, 1e6)), "targets": True}
        return {"kind": kind, "count": rng.randint(3, 10), "sizes": "40,64,96,130,160,192",
                "photons": int(_log_uniform(rng, 1e5, 5e5)), "targets": False}
    if kind == "layer":
        layer = rng.choice(["conv3", "conv3", "conv3", "down", "up"])
        edge = rng.choice([8, 16, 32, 64] if layer == "conv3" else [16, 32, 64] if layer == "down" else [8, 16, 32])
        D, H, W = edge, edge, edge
        if layer == "conv3" and edge >= 16 and rng.random() < 0.4:      # non-cubic crops
            D, H, W = (rng.choice([edge // 2, edge, edge]) for _ in range(3))
        c = {8: 256, 16: 128, 32: 64, 64: 32}[edge]
        c = rng.choice([c, c, c // 2, 16])
        if layer == "conv3":
            c0, c1, cout = rng.choice([(c, 0, c), (c, c, c), (16, 0, c)])
        elif layer == "down":
            c0, c1, cout = c, 0, min(256, 2 * c)
        else:
            c0, c1, cout = c, 0, max(16, c // 2)
        # multiply-adds of one direction log-uniform up to twice the listed layers'
        mac = D * H * W * TAPS[layer] * (c0 + c1) * cout / (8 if layer == "down" else 1)
        batch = min(max(1, int(_log_uniform(rng, 2e9, 2.5e11) / mac)), 5_000_000 // (D * H * W))
        if D * H * W < 4096:
            batch += batch % 2                  # 128-voxel tiles may span two samples
        return {"kind": kind, "layer": layer, "B": batch, "D": D, "H": H, "W": W, "c0": c0, "c1": c1, "cout": cout}
    c0, n = rng.choice([16, 32]), rng.choice([32, 64, 64])
    batch = max(1, int(_log_uniform(rng, 1, 48)))
    if n == 32:
        batch = 4 * batch                       # batch (n/8)^3 is a multiple of 128
    return {"kind": kind, "c0": c0, "n": n, "batch": batch}


# ----------------------------------------------------------------- prepare --

def _mask(shape, phi, seed):
    """Cahn-Hilliard mask (nz, ny, nx) made on the GPU; 512^3 is a periodic 64^3 field tiled."""
    nz, ny, nx = shape
    tile = 64 if min(shape) >= 512 and all(s % 64 == 0 for s in shape) else 0
    base = (tile,) * 3 if tile else shape
    steps = 1000 if base[0] * base[1] * base[2] <= 1 << 18 else 400
    c = inputs.cahn_hilliard(base, steps, seed=seed, device="cuda", dtype=torch.float32)
    m = inputs.rank_threshold(c, phi)
    return np.tile(m, (nz // tile, ny // tile, nx // tile)) if tile else m


def _batch_problems(case, seed):
    """Masks of the case's sizes in turn, porosity and optics distributed as in the batched
    configuration."""
    sizes = [int(s) for s in case["sizes"].split(",")]
    size = [sizes[i % len(sizes)] for i in range(case["count"])]
    rng = np.random.default_rng(seed)
    out = [None] * case["count"]
    for n in sorted(set(size)):
        idx = [i for i in range(case["count"]) if size[i] == n]
        c = inputs.cahn_hilliard((n,) * 3, 400, device="cuda", dtype=torch.float32, seeds=[1000 * seed + i for i in idx])
        for j, i in enumerate(idx):
            out[i] = (inputs.rank_threshold(c[j], float(rng.uniform(0.50, 0.95))),
                      float(np.exp(rng.uniform(math.log(0.1), math.log(2.0)))), float(rng.uniform(0.001, 0.05)),
                      float(rng.uniform(0.0, 0.9)))
    return out


def _net_inputs(case, seed):
    """Masks, optics and log-fluence-like targets of a network batch."""
    B, n = case["batch"], case["n"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    phi = torch.tensor(rng.uniform(0.50, 0.95, B), dtype=torch.float32, device="cuda")
    # smooth random phases: box-filtered noise, thresholded per sample to its porosity
    f = torch.randn((B, 1, n, n, n), generator=gen, device="cuda")
    for _ in range(2):
        f = torch.nn.functional.avg_pool3d(torch.nn.functional.pad(f, (2,) * 6, mode="circular"), 5, 1)
    flat = f.reshape(B, -1)
    rank = flat.argsort(dim=1).argsort(dim=1).float() / (n ** 3)
    mask = (rank >= 1.0 - phi[:, None]).to(torch.uint8).reshape(B, n, n, n).contiguous()
    optics = torch.tensor(np.stack([np.exp(rng.uniform(math.log(0.1), math.log(2.0), B)),
                                    rng.uniform(0.001, 0.05, B), rng.uniform(0.0, 0.9, B)], axis=1),
                          dtype=torch.float32, device="cuda")
    z = torch.arange(n, device="cuda", dtype=torch.float32).view(1, n, 1, 1) + 0.5
    slope = torch.tensor(rng.uniform(0.005, 0.08, B), dtype=torch.float32, device="cuda").view(B, 1, 1, 1)
    target = 0.4 - slope * z + 0.1 * torch.randn((B, n, n, n), generator=gen, device="cuda")
    return mask, optics, target.contiguous()


def _out_grid(case):
    B, D, H, W = case["B"], case["D"], case["H"], case["W"]
    return {"conv3": (B, D, H, W), "down": (B, D // 2, H // 2, W // 2), "up": (B, 2 * D, 2 * H, 2 * W)}[case["layer"]]


def _layer_tensors(case, seed):
    """Activations after a ReLU, output gradients, He-normal weights and small biases."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cin, cout, taps = case["c0"] + case["c1"], case["cout"], TAPS[case["layer"]]
    B, D, H, W = case["B"], case["D"], case["H"], case["W"]

    def planes(c, grid, relu):
        t = torch.randn((c // 8, *grid, 8), generator=gen, device="cuda")
        return (t.clamp_(min=0) if relu else t).to(torch.bfloat16)

    x0 = planes(case["c0"], (B, D, H, W), True)
    x1 = planes(case["c1"], (B, D, H, W), True) if case["c1"] else None
    dy = planes(cout, _out_grid(case), False)
    fan_in = cin if case["layer"] == "up" else taps * cin
    w = torch.randn((taps, cin, cout), generator=gen, device="cuda") * math.sqrt(2.0 / fan_in)
    b = torch.randn((cout,), generator=gen, device="cuda") * 0.1
    return x0, x1, dy, w, b


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed}
    if kind in ("mc", "noalloc"):
        mask = _mask((case["nz"], case["ny"], case["nx"]), case["phi"], seed)
        if kind == "noalloc":
            s["mask"] = torch.from_numpy(mask).cuda()
            return s
        s["sim"] = spmc.Simulation(mask, case["mu_s"], case["mu_a"], case["g"], precision=case["precision"],
                                   lateral_bc=case["mirror"], tally_field=int(case["tally"] == "field"))
        if case["tally"] == "field":
            s["fluence"] = torch.empty(mask.shape, dtype=torch.float32, device="cuda")
    elif kind == "batch":
        problems = _batch_problems(case, seed)
        s["batch"] = spmc.Batch(problems)
        s["fields"] = [torch.empty(p[0].shape, dtype=torch.int64, device="cuda") for p in problems]
        if case["targets"]:
            n = problems[0][0].shape[0]
            s["raw"] = torch.empty((case["count"], n, n, n), dtype=torch.int64, device="cuda")
            s["fields"] = list(s["raw"])
            s["n_photons"] = torch.full((case["count"],), float(case["photons"]), dtype=torch.float64, device="cuda")
            s["target"] = torch.empty((case["count"], n, n, n), dtype=torch.float32, device="cuda")
    elif kind == "layer":
        k, cin, cout = KINDS[case["layer"]], case["c0"] + case["c1"], case["cout"]
        s["x0"], s["x1"], s["dy"], w, s["b"] = _layer_tensors(case, seed)
        s["fwd"] = torch.empty(spnn.spnn_packed_elems(k, cin, cout), dtype=torch.bfloat16, device="cuda")
        s["bwd"] = torch.empty_like(s["fwd"])
        spnn.spnn_pack_weights(k, cin, cout, spnn.PACK_FWD, w, s["fwd"])
        spnn.spnn_pack_weights(k, cin, cout, spnn.PACK_DGRAD, w, s["bwd"])
        s["y"] = spnn.planes_empty(*_out_grid(case), cout)
        grid = (case["B"], case["D"], case["H"], case["W"])
        s["dx0"] = spnn.planes_empty(*grid, case["c0"])
        s["dx1"] = spnn.planes_empty(*grid, case["c1"]) if case["c1"] else None
        s["dw"], s["db"] = torch.empty_like(w), torch.empty_like(s["b"])
    else:
        B, n = case["batch"], case["n"]
        s["mask"], s["optics"], s["target"] = _net_inputs(case, seed)
        s["net"] = spnn.UNet(case["c0"], n, B)
        s["net"].set_params(spnn.init_params(case["c0"], seed))
        s["x"] = spnn.planes_empty(B, n, n, n, 16)
        s["pred"] = torch.empty((B, n, n, n), dtype=torch.float32, device="cuda")
        s["prof"] = torch.empty((B, 2, n), dtype=torch.float32, device="cuda")
    return s


# --------------------------------------------------------------------- run --

_INTS = ("launched", "interactions", "scatters", "rr_survive", "rr_kill", "exit_R", "exit_T", "gated_n", "steps",
         "solid_steps")
_RAW = ("raw_R", "raw_T", "raw_A", "raw_gated", "raw_lost", "raw_gain", "batch_photons", "raw_depth", "raw_hist",
        "raw_sum_w", "raw_sum_wP", "raw_sum_wP2", "depth_count")
_EST = ("R", "T", "A", "gated", "lost", "gain", "R_se", "T_se", "A_se", "phi_3d", "phi_1d", "phi_pore", "r", "ratio",
        "escape_weight", "pore_path_mean", "pore_path_m2", "p_pore_gt_L")


def _tallies(t):
    """The integer tallies, the event counts, the estimators and the depth profiles of a result."""
    return {"raw": np.concatenate([t[k].ravel() for k in _RAW]).view(np.int64),
            "events": np.array([t[k] for k in _INTS], dtype=np.int64),
            "estimators": np.array([t[k] for k in _EST]), "depth": t["depth"], "hist": t["pore_hist"]}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "noalloc":
        return _tallies(spmc.sp_mc_simulate_noalloc(s["mask"], case["nx"], case["ny"], case["nz"], 1.0, case["mu_s"],
                                                    case["mu_a"], case["g"], case["photons"], s["seed"]))
    if kind == "mc":
        sim = s["sim"]
        sim.reset()
        sim.run(case["photons"], s["seed"])
        out = _tallies(sim.tallies())
        if case["tally"] == "field":
            out["fluence"] = sim.fluence(s["fluence"])
        return out
    if kind == "batch":
        b = s["batch"]
        if case["targets"]:
            b.reset()
            b.run(case["photons"], s["seed"])
            for i, f in enumerate(s["fields"]):
                b.raw_field_to(i, f)
            spnn.spnn_log_fluence(s["raw"], s["n_photons"], s["target"])
            return {"raw": s["raw"], "target": s["target"]}
        b.run(case["photons"], s["seed"])           # further photons of the same problems
        for i, f in enumerate(s["fields"]):
            b.raw_field_to(i, f)
        t = [_tallies(b.tallies(i)) for i in range(case["count"])]
        return {"fields": s["fields"], **{k: np.stack([x[k] for x in t]) for k in t[0]}}
    if kind == "layer":
        k, cout = KINDS[case["layer"]], case["cout"]
        grid = (case["B"], case["D"], case["H"], case["W"])
        spnn.spnn_layer_forward(k, grid, s["x0"], s["x1"], s["fwd"], s["b"], cout, case["layer"] != "up", s["y"])
        # as in the network's backward: the gradient of a ReLU output is masked by it, the
        # two halves of a concatenated input are raw
        spnn.spnn_layer_dgrad(k, grid, s["dy"], s["bwd"], case["c0"], case["c1"], s["dx0"],
                              mask0=None if case["c1"] else s["x0"], dx1=s["dx1"])
        s["dw"].zero_()
        s["db"].zero_()
        spnn.spnn_layer_wgrad(k, grid, s["x0"], s["x1"], s["dy"], s["dw"], s["db"])
        return {"y": s["y"], "dx0": s["dx0"], "dx1": s["dx1"], "dw": s["dw"], "db": s["db"]}
    net = s["net"]
    spnn.spnn_pack_input(s["mask"], s["optics"], s["x"])
    net.forward(s["x"], s["pred"])
    if kind == "predict":
        spnn.spnn_phase_profiles(s["pred"], s["mask"], s["prof"])
        return {"pred": s["pred"], "profiles": s["prof"]}
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    net.backward(s["target"], loss)
    return {"pred": s["pred"], "loss": loss, "grads": net.get_grads()}


# -------------------------------------------------------------------- work --

def _steps_per_photon(case):
    """Voxel steps of a photon, roughly: a diffusive crossing of the slab takes about 3.5 nz
    (measured on the phi = 0.9 masks), an absorbing solid ends the history earlier."""
    phi = case.get("phi", 0.725)
    return min(3.5 * case["nz"], 20.0 + 1.5 * math.log(1e4) / max(1e-4, (1.0 - phi) * case["mu_a"]))


def _net_flops(c0, n, batch):
    level = {"e0": 0, "d1": 0, "e1": 1, "d2": 1, "e2": 2, "d3": 2, "b1": 3, "b2": 3, "u2": 3, "c2": 2, "u1": 2,
             "c1": 1, "u0": 1, "c0": 0}
    f = 0.0
    for name, kind, ci, co in spnn.layer_table(c0):
        vox = (n >> level[name[:2]]) ** 3
        taps = 27 if kind == "conv3" else 8
        f += 2.0 * taps * ci * co * (vox / 8 if kind == "down" else vox)
    return f * batch


def work(case):
    kind = case["kind"]
    if kind in ("mc", "noalloc"):
        vox = case["nx"] * case["ny"] * case["nz"]
        steps = case["photons"] * _steps_per_photon(case)
        field = kind == "mc" and case["tally"] == "field"
        # mask bits read, field and fluence written once; 37 lane operations per voxel step
        return {"bytes": vox / 8 + (12 * vox if field else 0) + (vox if kind == "noalloc" else 0), "flops": 37.0 * steps}
    if kind == "batch":
        sizes = [int(x) for x in case["sizes"].split(",")]
        sizes = [sizes[i % len(sizes)] for i in range(case["count"])]
        vox = sum(x ** 3 for x in sizes)
        nz = sum(sizes) / len(sizes)
        steps = case["count"] * case["photons"] * _steps_per_photon({"nz": nz, "mu_a": 0.02})
        return {"bytes": vox / 8 + 16 * vox + (4 * vox if case["targets"] else 0), "flops": 37.0 * steps}
    if kind == "layer":
        B, D, H, W = case["B"], case["D"], case["H"], case["W"]
        vin, cin, cout, taps = B * D * H * W, case["c0"] + case["c1"], case["cout"], TAPS[case["layer"]]
        Bo, Do, Ho, Wo = _out_grid(case)
        vout = Bo * Do * Ho * Wo
        mac = vout * taps if case["layer"] != "up" else vin * taps
        # x and dy read, y and dx written once each (BF16); FP32 weight gradient written, packed weights read
        return {"bytes": 4.0 * vin * cin + 4.0 * vout * cout + 8.0 * taps * cin * cout,
                "flops": 3 * 2.0 * mac * cin * cout}
    vox = case["batch"] * case["n"] ** 3
    params = sum((27 if k == "conv3" else 8) * ci * co for _, k, ci, co in spnn.layer_table(case["c0"]))
    f = _net_flops(case["c0"], case["n"], case["batch"])
    if kind == "predict":
        return {"bytes": vox * (1 + 4.0) + 2.0 * params, "flops": f}
    return {"bytes": vox * (1 + 4.0 + 4.0) + 6.0 * params, "flops": 3 * f}


# ------------------------------------------------------------------- exact --

def _voxels(planes):
    """Chunk planes (C/8, B, D, H, W, 8) -> FP64 (B, D, H, W, C)."""
    c8, B, D, H, W, _ = planes.shape
    return planes.permute(1, 2, 3, 4, 0, 5).reshape(B, D, H, W, 8 * c8).double()


def _planes(t):
    B, D, H, W, C = t.shape
    return t.reshape(B, D, H, W, C // 8, 8).permute(4, 0, 1, 2, 3, 5).contiguous()


def _offsets(kind):
    r = (-1, 0, 1) if kind == "conv3" else (0, 1)
    return [(z, y, x) for z in r for y in r for x in r]


def _shift(x, d):
    """x[v + d], zero outside (conv3 tap d)."""
    D, H, W = x.shape[1:4]
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    return p[:, 1 + d[0]:1 + d[0] + D, 1 + d[1]:1 + d[1] + H, 1 + d[2]:1 + d[2] + W]


def _layer64(kind, x, w, b):
    """One layer in FP64: x (B, D, H, W, cin), w [taps][cin][cout]."""
    B, D, H, W, _ = x.shape
    if kind == "conv3":
        return sum(_shift(x, d) @ w[t] for t, d in enumerate(_offsets(kind))) + b
    if kind == "down":
        return sum(x[:, d[0]::2, d[1]::2, d[2]::2] @ w[t] for t, d in enumerate(_offsets(kind))) + b
    y = torch.empty((B, 2 * D, 2 * H, 2 * W, w.shape[2]), dtype=torch.float64, device=x.device)
    for t, d in enumerate(_offsets(kind)):
        y[:, d[0]::2, d[1]::2, d[2]::2] = x @ w[t] + b
    return y


def _exact_layer(case, seed):
    x0, x1, dy, w, b = _layer_tensors(case, seed)
    kind = case["layer"]
    x = torch.cat([_voxels(x0)] + ([_voxels(x1)] if x1 is not None else []), dim=-1)
    w, b, g = w.to(torch.bfloat16).double(), b.double(), _voxels(dy)
    y = _layer64(kind, x, w, b)
    if kind != "up":
        y = y.clamp(min=0)
    dx, dw = torch.zeros_like(x), torch.empty_like(w)
    ci, co = w.shape[1:]
    for t, d in enumerate(_offsets(kind)):
        if kind == "conv3":
            dx += _shift(g, tuple(-k for k in d)) @ w[t].T
            dw[t] = _shift(x, d).reshape(-1, ci).T @ g.reshape(-1, co)
        else:
            v = (slice(None), slice(d[0], None, 2), slice(d[1], None, 2), slice(d[2], None, 2))
            if kind == "down":
                dx[v] = g @ w[t].T
                dw[t] = x[v].reshape(-1, ci).T @ g.reshape(-1, co)
            else:
                dx += g[v] @ w[t].T
                dw[t] = x.reshape(-1, ci).T @ g[v].reshape(-1, co)
    if not case["c1"]:
        dx = dx * (x > 0)
    c0 = case["c0"]
    return {"y": _planes(y), "dx0": _planes(dx[..., :c0]), "dx1": _planes(dx[..., c0:]) if case["c1"] else None,
            "dw": dw, "db": g.reshape(-1, co).sum(0)}


def _exact_predict(case, seed):
    mask, optics, _ = _net_inputs(case, seed)
    B, n, c0 = case["batch"], case["n"], case["c0"]
    pore = mask.double()
    phi = pore.mean(dim=(1, 2, 3))
    mus, mua, g = optics.double().unbind(1)
    ma, msp = (1 - phi) * mua, (1 - phi) * mus * (1 - g)
    mu_eff = torch.sqrt(3 * ma * (ma + msp))
    zc = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5
    x = torch.zeros((B, n, n, n, 16), dtype=torch.float64, device="cuda")
    x[..., 0], x[..., 1] = pore, 1 - pore
    for i, v in ((2, torch.log(mus)), (3, torch.log(mua) / 4), (4, g), (7, phi)):
        x[..., i] = v.view(B, 1, 1, 1)
    x[..., 5] = (zc / n).view(1, n, 1, 1)
    x[..., 6] = -mu_eff.view(B, 1, 1, 1) * zc.view(1, n, 1, 1) / 8
    flat = torch.from_numpy(spnn.init_params(c0, seed)).cuda().double()
    off, acts = 0, []
    for i, (name, kind, ci, co) in enumerate(spnn.layer_table(c0)):
        taps = TAPS[kind]
        w = flat[off:off + taps * ci * co].reshape(taps, ci, co)
        off += taps * ci * co
        b = flat[off:off + co]
        off += co
        skip = {"c2a": 7, "c1a": 4, "c0a": 1}.get(name)
        h = x if i == 0 else acts[-1]
        if skip is not None:
            h = torch.cat([h, acts[skip]], dim=-1)
        y = _layer64(kind, h, w, b)
        acts.append(y if kind == "up" else y.clamp(min=0))
    pred = acts[-1] @ flat[off:off + c0] + flat[off + c0]
    e = torch.exp(pred)
    prof = torch.stack([(e * m).sum(dim=(2, 3)) / m.sum(dim=(2, 3)) for m in (1 - pore, pore)], dim=1)
    return {"pred": pred, "profiles": prof}


def exact(case, seed):
    """FP64 outputs of a layer, or of a small network batch.  A photon run has none: its integer
    tallies are compared as they are, and its estimators follow from them."""
    if case["kind"] == "layer":
        macs = case["B"] * case["D"] * case["H"] * case["W"] * TAPS[case["layer"]] * (case["c0"] + case["c1"]) * case["cout"]
        return _exact_layer(case, seed) if macs <= 6e11 else None
    if case["kind"] == "predict" and case["batch"] * (case["n"] / 64) ** 3 <= 2:
        return _exact_predict(case, seed)
    return None

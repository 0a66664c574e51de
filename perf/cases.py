"""The work this framework is used for, as cases that a timing program can run.

A case is one call (or one training step) as a program makes it through the
package's public entry points: an image of a transducer's field through one
interface, through a laminate, on both sides of an interface, by the
ray-tracing model, of a focused transducer, of several frequencies at once, a
batched scan, and the learned surrogate's training step and inference.
`listed()` holds the sizes of the package's own workloads (workloads.py),
`draw()` others of the same ranges, `prepare()` what a program holds before the
call, `run()` the call, `work()` what the call cannot do without and `exact()`
the result in 64 bits by plain torch and numpy.

FP32C images are taken as complex64, the format their accuracy (about 1e-6)
fills; FP64 images as complex128.
"""
from __future__ import annotations

import cmath
import math

import numpy as np
import torch

from paper_2408_06765_gb300 import rsi
from paper_2408_06765_gb300 import surrogate as S
from paper_2408_06765_gb300 import workloads as W

MM = 1e-3
MHZ = 1e6


def listed() -> list[dict]:
    return [
        # the smallest call: one field image of a few hundred pixels, as in an
        # interactive set-up or an optimiser's inner loop; ragged counts
        {"name": "chain_small", "kind": "chain", "precision": "fp32c", "freq": 5.0, "tilt": 0.0, "z_if": 30.0,
         "patch": 40.0, "half": 15.0, "depth": 25.0, "n_piston": 1000, "n_iface": 3000, "nx": 37, "nz": 29},
        # the validation run: plain RSI in FP64 (c1)
        {"name": "chain_fp64", "kind": "chain", "precision": "fp64", "freq": 5.0, "tilt": 0.0, "z_if": 50.0,
         "patch": 60.0, "half": 20.0, "depth": 40.0, "n_piston": 4096, "n_iface": 4096, "nx": 64, "nz": 64},
        # an ordinary field: a tilted transducer at the surrogate's first point counts
        {"name": "chain_tilted", "kind": "chain", "precision": "fp32c", "freq": 4.0, "tilt": 8.0, "z_if": 40.0,
         "patch": 60.0, "half": 20.0, "depth": 40.0, "n_piston": 16384, "n_iface": 65536, "nx": 128, "nz": 128},
        # the full image at three frequencies on shared points (c2): the largest
        {"name": "image_multi", "kind": "multi", "freqs": "2.25 5 10", "z_if": 50.0, "patch": 80.0, "half": 40.0,
         "depth": 60.0, "n_piston": 65536, "n_iface": 262144, "nx": 512, "nz": 512},
        # the laminate of eight layers, flat and curved (c3)
        {"name": "layers_flat", "kind": "layers", "curved": False, "freq": 5.0, "n": 65536, "nx": 256, "nz": 256},
        {"name": "layers_curved", "kind": "layers", "curved": True, "freq": 5.0, "n": 65536, "nx": 256, "nz": 256},
        # incident + reflected field above and transmitted field below an interface (f1)
        {"name": "two_medium", "kind": "two_medium", "freq": 5.0, "tilt": 10.0, "n_piston": 65536,
         "n_iface": 262144, "nx": 512, "nz": 256},
        # the ray-tracing model on the full image (f2)
        {"name": "raytrace", "kind": "raytrace", "freq": 5.0, "tilt": 10.0, "n_piston": 65536, "nx": 512,
         "nz": 512},
        # a focused transducer (f4) at a survey resolution
        {"name": "focused", "kind": "focused", "freq": 2.5, "n_piston": 16384, "n_iface": 65536, "nx": 256,
         "nz": 256},
        # a scan of positions and frequencies with uneven point counts in one graph (c4)
        {"name": "scan", "kind": "scan", "n_inst": 64, "log2_lo": 12, "log2_hi": 16, "nx": 128, "nz": 128},
        # one training step of the surrogate, replayed from a graph, and images of its network
        {"name": "train", "kind": "train", "rows": 32768, "width": 512, "depth": 5, "fields": 24},
        {"name": "infer", "kind": "infer", "rows": 65536, "width": 512, "depth": 5, "fields": 64},
    ]


def _log(rng, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["chain", "chain", "fp64", "multi", "layers", "two_medium", "raytrace", "focused", "scan",
                       "train", "infer"])
    if kind == "chain":
        return {"kind": "chain", "precision": "fp32c", "freq": rng.uniform(2.0, 7.0), "tilt": rng.uniform(-9.0, 9.0),
                "z_if": rng.uniform(20.0, 60.0), "patch": rng.uniform(40.0, 80.0), "half": rng.uniform(10.0, 40.0),
                "depth": rng.uniform(20.0, 60.0), "n_piston": _log(rng, 1000, 65536),
                "n_iface": _log(rng, 3000, 262144), "nx": _log(rng, 24, 512), "nz": _log(rng, 24, 512)}
    if kind == "fp64":
        return {"kind": "chain", "precision": "fp64", "freq": rng.uniform(2.0, 10.0), "tilt": rng.uniform(-9.0, 9.0),
                "z_if": rng.uniform(20.0, 60.0), "patch": rng.uniform(40.0, 80.0), "half": rng.uniform(10.0, 30.0),
                "depth": rng.uniform(20.0, 60.0), "n_piston": _log(rng, 500, 8192), "n_iface": _log(rng, 1000, 16384),
                "nx": _log(rng, 24, 128), "nz": _log(rng, 24, 128)}
    if kind == "multi":
        f = [round(rng.uniform(1.0, 5.0), 3) for _ in range(rng.randint(2, 3))]
        if len(f) == 2 or rng.random() < 0.5:
            f = f[:2] + [2.0 * f[1]]  # a harmonic, as in 2.25, 5 and 10 MHz
        return {"kind": "multi", "freqs": " ".join(str(v) for v in f), "z_if": rng.uniform(20.0, 60.0),
                "patch": rng.uniform(40.0, 80.0), "half": rng.uniform(10.0, 40.0), "depth": rng.uniform(20.0, 60.0),
                "n_piston": _log(rng, 4096, 65536), "n_iface": _log(rng, 16384, 262144), "nx": _log(rng, 64, 512),
                "nz": _log(rng, 64, 512)}
    if kind == "layers":
        return {"kind": "layers", "curved": rng.random() < 0.5, "freq": rng.uniform(2.0, 5.0),
                "n": _log(rng, 16384, 65536), "nx": _log(rng, 64, 256), "nz": _log(rng, 64, 256)}
    if kind == "two_medium":
        return {"kind": "two_medium", "freq": rng.uniform(2.0, 6.0), "tilt": rng.uniform(-12.0, 12.0),
                "n_piston": _log(rng, 4096, 65536), "n_iface": _log(rng, 16384, 262144), "nx": _log(rng, 64, 512),
                "nz": 2 * _log(rng, 16, 128)}  # the second window's image starts on 16 bytes
    if kind == "raytrace":
        return {"kind": "raytrace", "freq": rng.uniform(2.0, 10.0), "tilt": rng.uniform(-12.0, 12.0),
                "n_piston": _log(rng, 1000, 65536), "nx": _log(rng, 32, 512), "nz": _log(rng, 32, 512)}
    if kind == "focused":
        return {"kind": "focused", "freq": rng.uniform(1.5, 5.0), "n_piston": _log(rng, 2048, 65536),
                "n_iface": _log(rng, 8192, 262144), "nx": _log(rng, 32, 512), "nz": _log(rng, 32, 512)}
    if kind == "scan":
        return {"kind": "scan", "n_inst": _log(rng, 4, 96), "log2_lo": 12, "log2_hi": rng.choice([14, 15, 16]),
                "nx": _log(rng, 48, 160), "nz": _log(rng, 48, 160)}
    if kind == "train":
        return {"kind": "train", "rows": 128 * _log(rng, 32, 512), "width": rng.choice([256, 512]),
                "depth": rng.randint(2, 6), "fields": rng.randint(4, 32)}
    return {"kind": "infer", "rows": 16384 * rng.randint(1, 4), "width": rng.choice([256, 512]),
            "depth": rng.randint(2, 6), "fields": _log(rng, 1, 128)}


# ---------------------------------------------------------------------------
# workload descriptions
# ---------------------------------------------------------------------------
def _chain_cfg(case: dict, freq: float, seed: int) -> dict:
    tilt = math.radians(case.get("tilt", 0.0))
    zi, h = case["z_if"] * MM, case["half"] * MM
    xc = zi * math.tan(tilt)  # where the transducer axis meets the interface
    return {"name": "chain", "freq": freq * MHZ, "v0": 1.0, "seed": seed, "precision": case.get("precision", "fp32c"),
            "piston": {"a": 6.35 * MM, "centre": (0.0, 0.0, 0.0), "tilt": tilt, "n": case["n_piston"], "set_id": 0},
            "media": [dict(W.WATER), dict(W.STEEL)],
            "interfaces": [{"kind": "rect", "centre": (xc, 0.0, zi), "wx": case["patch"] * MM,
                            "wy": case["patch"] * MM, "n": case["n_iface"], "set_id": 1}],
            "tmode": "global",
            "grid": {"x0": xc - h, "x1": xc + h, "nx": case["nx"], "z0": zi, "z1": zi + case["depth"] * MM,
                     "nz": case["nz"], "y": 0.0}}


def _cfgs(case: dict, seed: int) -> list[dict]:
    kind = case["kind"]
    if kind == "chain":
        return [_chain_cfg(case, case["freq"], seed)]
    if kind == "multi":
        return [_chain_cfg(case, float(f), seed) for f in case["freqs"].split()]
    if kind == "layers":
        cfg = W.c3_multilayer(case["curved"], case["n"])
        cfg["freq"] = case["freq"] * MHZ
        cfg["grid"].update({"nx": case["nx"], "nz": case["nz"]})
    elif kind == "two_medium":
        cfg = W.f1_two_medium(case["freq"] * MHZ, case["tilt"], case["n_piston"], case["n_iface"], case["nx"],
                              case["nz"], case["nz"])
    elif kind == "raytrace":
        cfg = W.f2_ray_tracing(case["freq"] * MHZ, case["tilt"], case["n_piston"], case["nx"], case["nz"])
    elif kind == "focused":
        cfg = W.f4_focused(case["freq"] * MHZ, case["n_piston"], case["n_iface"], case["nx"], case["nz"])
    else:  # scan: frequencies and positions of c4, counts log-uniform
        gen = np.random.default_rng(seed)
        u = gen.random((case["n_inst"], 2))
        lo, hi = case["log2_lo"], case["log2_hi"]
        counts = np.rint(np.exp2(lo + (hi - lo) * u)).astype(np.int64)
        out = []
        for i in range(case["n_inst"]):
            jf, pos = int(gen.integers(0, W.C4_NFREQ)), int(gen.integers(0, W.C4_NPOS))
            full = np.zeros((W.C4_NFREQ * W.C4_NPOS, 2), np.int64)
            full[jf * W.C4_NPOS + pos] = counts[i]
            c = W.c4_instance(jf, pos, full)
            c["piston"]["set_id"], c["interfaces"][0]["set_id"] = 2 * i, 2 * i + 1
            c["seed"] = seed
            c["grid"].update({"nx": case["nx"], "nz": case["nz"]})
            out.append(c)
        return out
    cfg["seed"] = seed
    return [cfg]


def _net(case: dict, seed: int) -> S.CoordNet:
    return S.CoordNet(width=case["width"], depth=case["depth"], rows=case["rows"], seed=seed)


def _params(n: int, seed: int) -> np.ndarray:
    p = W.c5_params(n, seed)
    p[:, 1] *= 13.0 / 15.0  # the tilts the surrogate is trained on
    return p


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind == "train":
        net = _net(case, seed)
        p = _params(case["fields"], seed)
        imgs = S.rsi_images(p, n_piston=1 << 12, n_iface=1 << 14)
        tset = S.TrainingSet(net, p, imgs)
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        net.hyper.copy_(torch.tensor([1e-3, 1.0 - b1, 1.0 - b2]))
        net.rows_random(tset.params, tset.targets, tset.log_rms, seed=seed + 1)
        net.forward()
        net.backward()
        net.adam()
        net.step_count += 1
        seeds = np.random.default_rng(seed + 2).integers(0, 2**62, size=20000, dtype=np.int64)
        torch.cuda.synchronize()
        return {"net": net, "trainer": S.GraphedTrainer(net, tset, [1e-3] * 20000, seeds), "tset": tset,
                "seeds": seeds, "kind": kind}
    if kind == "infer":
        net = _net(case, seed)
        return {"net": net, "params": torch.tensor(_params(case["fields"], seed), device="cuda"), "kind": kind}
    cfgs = _cfgs(case, seed)
    if kind == "scan":
        return {"batch": rsi.Batch(cfgs, seed=seed), "kind": kind}
    return {"cfgs": cfgs, "ws": rsi.Workspace(), "kind": kind,
            "fmt": "c128" if case.get("precision") == "fp64" else "c64"}


def run(state: dict):
    kind = state["kind"]
    if kind == "train":
        loss = state["trainer"].step()
        net = state["net"]
        return {"loss": loss, "grad": net.g, "weights": net.w}
    if kind == "infer":
        return state["net"].infer(state["params"])
    if kind == "scan":
        return state["batch"].run()
    cfgs, ws, fmt = state["cfgs"], state["ws"], state["fmt"]
    if kind == "multi":
        return rsi.run_chain_multi(cfgs, fmt=fmt, workspace=ws)
    if kind == "two_medium":
        return rsi.run_two_medium(cfgs[0], fmt=fmt, workspace=ws).image
    if kind == "raytrace":
        return rsi.run_raytrace(cfgs[0], fmt=fmt, workspace=ws)
    return rsi.run_chain(cfgs[0], fmt=fmt, workspace=ws).image


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _pairs(case: dict) -> int:
    kind = case["kind"]
    if kind == "raytrace":
        return case["n_piston"] * case["nx"] * case["nz"]
    if kind == "two_medium":
        return rsi.two_medium_pairs(_cfgs(case, 0)[0])
    return sum(W.pairs_of(c) for c in _cfgs(case, 0))


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("train", "infer"):
        w, d, k0 = case["width"], case["depth"], 2 * 248 + 16
        params = w * k0 + (d - 1) * w * w + d * w + 3 * w + 3
        if kind == "train":
            # weights, moments read and written, the bf16 copy; 3 GEMMs per weight but the first's input gradient
            return {"bytes": 30 * params + 8 * case["rows"], "flops": 2 * case["rows"] * (3 * params - w * k0)}
        n = case["fields"] * S.NPIX
        return {"bytes": 2 * params + 8 * n + 40 * case["fields"], "flops": 2 * n * params}
    # inputs are scalars: the image is what has to be written; a pair term is
    # about 20 operations (distance, reciprocal, sine, cosine, products)
    size = 16 if case.get("precision") == "fp64" else 8
    cfgs = _cfgs(case, 0)
    if kind == "two_medium":
        pix = case["nx"] * 2 * case["nz"]
    else:
        pix = sum(int(c["grid"]["nx"]) * int(c["grid"]["nz"]) for c in cfgs)
    return {"bytes": size * pix, "flops": (60 if kind == "raytrace" else 20) * _pairs(case)}


# ---------------------------------------------------------------------------
# the result in 64 bits
# ---------------------------------------------------------------------------
EXACT_PAIRS = 1.2e10  # about 15 seconds of torch in FP64
EXACT_RAYS = 6e8


def _mix(z: np.ndarray) -> np.ndarray:
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


_GAMMA = np.uint64(0x9E3779B97F4A7C15)


def _sobol(seed: int, set_id: int, n: int):
    """(u, v) of the scrambled Sobol points 0 .. n-1 of a set."""
    with np.errstate(over="ignore"):
        i = np.arange(n, dtype=np.uint64)
        x = np.zeros(n, np.uint64)
        y = np.zeros(n, np.uint64)
        m = 1
        for j in range(1, 33):
            if j > 1:
                m = ((m << 1) ^ m) & 0xFFFFFFFF
            bit = (i >> np.uint64(j - 1)) & np.uint64(1)
            x ^= bit << np.uint64(32 - j)
            y ^= bit * np.uint64((m << (32 - j)) & 0xFFFFFFFF)
        base = _mix(np.array([seed], np.uint64) + _GAMMA)
        out = []
        for dim, w in enumerate((x, y)):
            key = _mix(base ^ np.uint64((set_id << 1) | dim))
            flips = np.zeros(n, np.uint64)
            for b in range(32):
                node = np.uint64(1 << b) | (w >> np.uint64(32 - b) if b else np.uint64(0))
                flips |= (_mix(key + node * _GAMMA) >> np.uint64(63)) << np.uint64(31 - b)
            out.append(((w ^ flips).astype(np.float64) + 0.5) * 2.0**-32)
    return out


def _surface(s: dict, seed: int):
    """Points (n, 3), normals (n, 3) and weights (n) of a surface, FP64 on the GPU."""
    n, kind = int(s["n"]), s.get("kind", "disk")
    u, v = (torch.tensor(a, device="cuda") for a in _sobol(seed, int(s.get("set_id", 0)), n))
    cx, cy, cz = s["centre"]
    one = torch.ones_like(u)
    if kind in ("disk", "cap"):
        t, a = float(s.get("tilt", 0.0)), s["a"]
        r = a * u.sqrt()
        l1, l2 = r * torch.cos(2 * math.pi * v), r * torch.sin(2 * math.pi * v)
        w = math.pi * a * a / n * one
        h, n1, n2, n3 = 0 * one, 0 * one, 0 * one, one
        if kind == "cap":
            q = (s["R"] ** 2 - r * r).sqrt()
            h, n1, n2, n3, w = s["R"] - q, -l1 / s["R"], -l2 / s["R"], q / s["R"], w * s["R"] / q
        ct, st = math.cos(t), math.sin(t)
        P = torch.stack([cx + l1 * ct + h * st, cy + l2, cz - l1 * st + h * ct], 1)
        N = torch.stack([n1 * ct + n3 * st, n2, -n1 * st + n3 * ct], 1)
        return P, N, w
    xi, yi = s["wx"] * (u - 0.5), s["wy"] * (v - 0.5)
    w = s["wx"] * s["wy"] / n * one
    if kind == "cyl":
        q = (s["R"] ** 2 - xi * xi).sqrt()
        return (torch.stack([cx + xi, cy + yi, cz + s["R"] - q], 1), torch.stack([-xi / s["R"], 0 * xi, q / s["R"]], 1),
                w * s["R"] / q)
    return torch.stack([cx + xi, cy + yi, cz * one], 1), torch.stack([0 * one, 0 * one, one], 1), w


def _grid(g: dict) -> torch.Tensor:
    x = g["x0"] + (torch.arange(g["nx"], dtype=torch.float64, device="cuda") + 0.5) * ((g["x1"] - g["x0"]) / g["nx"])
    z = g["z0"] + (torch.arange(g["nz"], dtype=torch.float64, device="cuda") + 0.5) * ((g["z1"] - g["z0"]) / g["nz"])
    Z, X = torch.meshgrid(z, x, indexing="ij")
    return torch.stack([X.reshape(-1), torch.full_like(X, g.get("y", 0.0)).reshape(-1), Z.reshape(-1)], 1)


def _stage(Q, P, N, w, sigma, k: float, v0: float) -> torch.Tensor:
    """The piston sum (sigma None) or the Rayleigh-Sommerfeld sum at the targets Q."""
    out = torch.empty(len(Q), dtype=torch.complex128, device=Q.device)
    step = max(1, (1 << 25) // len(P))
    for a in range(0, len(Q), step):
        q = Q[a:a + step]
        d = [q[:, None, c] - P[None, :, c] for c in range(3)]
        r = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).sqrt()
        kr = k * r
        cs, sn = torch.cos(kr), torch.sin(kr)
        if sigma is None:
            A = (-v0 / (2 * math.pi)) * w / r
            re, im = (A * cs).sum(1), (A * sn).sum(1)
        else:
            h = (N[:, 0] * d[0] + N[:, 1] * d[1] + N[:, 2] * d[2]) / (r * r)
            Br, Bi = -w * sigma.real / (2 * math.pi), -w * sigma.imag / (2 * math.pi)
            vr, vi = -Br / r - k * Bi, -Bi / r + k * Br
            re, im = (h * (vr * cs - vi * sn)).sum(1), (h * (vr * sn + vi * cs)).sum(1)
        out[a:a + step] = torch.complex(re, im)
    return out


def _cosines(cfg: dict, s: int, N):
    """cos of the incidence and refraction angles at interface s (global or local mode)."""
    C = math.sin(cfg["piston"].get("tilt", 0.0)) / cfg["media"][0]["c"]
    c1, c2 = cfg["media"][s]["c"], cfg["media"][s + 1]["c"]
    if cfg.get("tmode", "global") == "global":
        return cmath.sqrt(1 - (c1 * C) ** 2), cmath.sqrt(1 - (c2 * C) ** 2)
    s1 = c1 * C
    a = (s1 * N[:, 0] + math.sqrt(max(0.0, 1 - s1 * s1)) * N[:, 2]).clamp(0.0, 1.0)
    return a, torch.sqrt(torch.complex(1 - (c2 / c1) ** 2 * (1 - a * a), torch.zeros_like(a)))


def _t12(cfg: dict, s: int, N):
    m1, m2 = cfg["media"][s], cfg["media"][s + 1]
    a1, a2 = _cosines(cfg, s, N)
    return 2 * m1["rho"] * m2["c"] * a1 / (m2["rho"] * m2["c"] * a1 + m1["rho"] * m1["c"] * a2)


def _r12(cfg: dict, s: int, N):
    m1, m2 = cfg["media"][s], cfg["media"][s + 1]
    a1, a2 = _cosines(cfg, s, N)
    return ((m2["rho"] * m2["c"] * a1 - m1["rho"] * m1["c"] * a2) /
            (m2["rho"] * m2["c"] * a1 + m1["rho"] * m1["c"] * a2))


def _image(cfg: dict, seed: int) -> torch.Tensor:
    k = [2 * math.pi * cfg["freq"] / m["c"] for m in cfg["media"]]
    P, N, w = _surface(cfg["piston"], seed)
    sigma, v0 = None, cfg["v0"]
    for s, it in enumerate(cfg["interfaces"]):
        P2, N2, w2 = _surface(it, seed)
        phi = _stage(P2, P, N, w, sigma, k[s], v0)
        P, N, w, sigma = P2, N2, w2, phi * _t12(cfg, s, N2)
    g = cfg["grid"]
    return (k[-1] / v0 * _stage(_grid(g), P, N, w, sigma, k[-1], v0)).view(g["nz"], g["nx"])


def _two_medium(cfg: dict, seed: int) -> torch.Tensor:
    k = [2 * math.pi * cfg["freq"] / m["c"] for m in cfg["media"]]
    P, N, w = _surface(cfg["piston"], seed)
    I, NI, wi = _surface(cfg["interfaces"][0], seed)
    gw, gs, v0 = cfg["grid_water"], cfg["grid_solid"], cfg["v0"]
    phi = _stage(I, P, N, w, None, k[0], v0)
    Qw, Qs = _grid(gw), _grid(gs)
    up = _stage(Qw, P, N, w, None, k[0], v0) + _stage(Qw, I, -NI, wi, phi * _r12(cfg, 0, NI), k[0], v0)
    down = _stage(Qs, I, NI, wi, phi * _t12(cfg, 0, NI), k[1], v0)
    return torch.cat([(k[0] / v0 * up).view(gw["nz"], gw["nx"]), (k[1] / v0 * down).view(gs["nz"], gs["nx"])])


def _rays(cfg: dict, seed: int) -> torch.Tensor:
    m1, m2 = cfg["media"]
    c1, c2, zi, v0, g = m1["c"], m2["c"], cfg["interfaces"][0]["centre"][2], cfg["v0"], cfg["grid"]
    k1, k2 = 2 * math.pi * cfg["freq"] / c1, 2 * math.pi * cfg["freq"] / c2
    P, _, w = _surface(cfg["piston"], seed)
    Q = _grid(g)
    out = torch.empty(len(Q), dtype=torch.complex128, device=Q.device)
    step = max(1, (1 << 24) // len(P))
    for a in range(0, len(Q), step):
        q = Q[a:a + step]
        rho = ((q[:, None, 0] - P[None, :, 0]) ** 2 + (q[:, None, 1] - P[None, :, 1]) ** 2).sqrt()
        h1, h2 = (zi - P[:, 2])[None, :].expand_as(rho), (q[:, 2] - zi)[:, None].expand_as(rho)
        lo, hi = torch.zeros_like(rho), rho.clone()
        t = rho * h1 / (h1 + c2 / c1 * h2)
        for _ in range(60):  # Newton inside a bracket of Snell's monotone residual
            D1, D2 = (t * t + h1 * h1).sqrt(), ((rho - t) ** 2 + h2 * h2).sqrt()
            G = t / (c1 * D1) - (rho - t) / (c2 * D2)
            hi, lo = torch.where(G > 0, t, hi), torch.where(G > 0, lo, t)
            tn = t - G / (h1 * h1 / (c1 * D1**3) + h2 * h2 / (c2 * D2**3))
            tn = torch.where((tn >= lo) & (tn <= hi), tn, 0.5 * (lo + hi))
            if float((tn - t).abs().max()) < 1e-16:
                break
            t = tn
        D1, D2 = (t * t + h1 * h1).sqrt(), ((rho - t) ** 2 + h2 * h2).sqrt()
        a1, a2 = h1 / D1, h2 / D2
        T = 2 * m1["rho"] * c2 * a1 / (m2["rho"] * c2 * a1 + m1["rho"] * c1 * a2)
        den = ((D1 + c2 * a1 * a1 / (c1 * a2 * a2) * D2) * (D1 + c2 / c1 * D2)).sqrt()
        A, ph = -v0 / (2 * math.pi) * w * T / den, k1 * D1 + k2 * D2
        out[a:a + step] = torch.complex((A * torch.cos(ph)).sum(1), (A * torch.sin(ph)).sum(1))
    return (k2 / v0 * out).view(g["nz"], g["nx"])


def _net_rows(net: S.CoordNet, p: torch.Tensor, q: torch.Tensor) -> torch.Tensor:
    """Inputs (rows, 2F + 16) of the network for parameter rows p and pixels q."""
    nx, win = S.WINDOW["nx"], S.WINDOW
    dx, dz = (win["x1"] - win["x0"]) / nx, (win["z1"] - win["z0"]) / win["nz"]
    xw, zw = win["x0"] + (q % nx + 0.5) * dx, win["z0"] + (q // nx + 0.5) * dz
    tilt, L, f, d = p[:, 1], p[:, 2], p[:, 3], p[:, 4]
    sg, a1 = torch.where(tilt < 0, -1.0, 1.0).double(), tilt.abs()
    x, z, c21 = sg * xw, d + zw, S.C2 / S.C1
    sth = (c21 * a1.sin()).clamp(max=1.0)
    cth = (1 - sth * sth).clamp(min=0.0).sqrt()
    s, t = x * sth + z * cth, x * cth - z * sth
    fq = S.A_PISTON**2 / S.C1 * f / (L + c21 * s.clamp(min=0.0))
    nrm = [2 * (v - lo) / (hi - lo) - 1 for v, lo, hi in zip((a1, L, f, d), S.BOX_LO, S.BOX_HI)]
    s0 = (win["x1"] - win["x0"]) / 2
    c = torch.stack(nrm + [x / s0, 2 * (zw - win["z0"]) / (win["z1"] - win["z0"]) - 1, s / s0, t / s0, fq.log()], 1)
    arg = math.pi * (c @ net.fmat.double().T)
    return torch.cat([arg.sin(), arg.cos(), c, torch.zeros(len(c), 7, dtype=c.dtype, device=c.device)], 1)


def _net_forward(net: S.CoordNet, h: torch.Tensor, w: torch.Tensor) -> torch.Tensor:
    for l in range(net.depth + 1):
        h = torch.nn.functional.linear(h, net.layer(l, False, w), net.layer(l, True, w))
        if l < net.depth:
            h = torch.nn.functional.silu(h)
    return h


def _infer(state: dict) -> torch.Tensor:
    net, p = state["net"], state["params"].double()
    q = torch.arange(S.NPIX, device="cuda")
    ys = []
    for i in range(len(p)):
        ys.append(_net_forward(net, _net_rows(net, p[i:i + 1].expand(S.NPIX, -1), q), net.w.double()))
    y = torch.stack(ys)
    nx, win = S.WINDOW["nx"], S.WINDOW
    dx, dz = (win["x1"] - win["x0"]) / nx, (win["z1"] - win["z0"]) / win["nz"]
    xw, zw = win["x0"] + (q % nx + 0.5) * dx, win["z0"] + (q // nx + 0.5) * dz
    s = S.C2 / S.C1 * p[:, 1].sin()
    c = (1 - s * s).clamp(min=0.0).sqrt()
    k1, k2 = 2 * math.pi * p[:, 3] / S.C1, 2 * math.pi * p[:, 3] / S.C2
    psi = (k1 * p[:, 2])[:, None] + k2[:, None] * (s[:, None] * xw + c[:, None] * (p[:, 4][:, None] + zw))
    amp = y[:, :, 2].mean(1, keepdim=True).exp()
    img = torch.complex(amp * y[:, :, 0], amp * y[:, :, 1]) * torch.polar(torch.ones_like(psi), psi)
    return img.view(len(p), win["nz"], nx)


def _train(state: dict, case: dict) -> dict:
    net, tset = state["net"], state["tset"]
    R, n = case["rows"], tset.params.shape[0]
    with np.errstate(over="ignore"):
        u = _mix(np.array([state["seeds"][0]], np.uint64) + _GAMMA * np.arange(1, R + 1, dtype=np.uint64))
        b = ((u >> np.uint64(32)) * np.uint64(n)) >> np.uint64(32)
        q = ((u & np.uint64(0xFFFFFFFF)) * np.uint64(S.NPIX)) >> np.uint64(32)
    b, q = (torch.tensor(v.astype(np.int64), device="cuda") for v in (b, q))
    t = torch.cat([tset.targets.double().view(n, S.NPIX, 2)[b, q], tset.log_rms.double()[b][:, None]], 1)
    w = net.w.double().clone().requires_grad_(True)
    loss = ((_net_forward(net, _net_rows(net, tset.params[b], q), w) - t) ** 2).sum() / (4.0 * R)
    loss.backward()
    g = w.grad
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))  # this is the second step
    m, v = b1 * net.m.double() + (1 - b1) * g, b2 * net.v.double() + (1 - b2) * g * g
    new = w.detach() - 1e-3 * (m / (1 - b1**2)) / ((v / (1 - b2**2)).sqrt() + 1e-8)
    return {"loss": loss.detach().view(1), "grad": g, "weights": new}


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "infer":
        return _infer(prepare(case, seed)) if case["fields"] * S.NPIX * case["depth"] <= 6e6 else None
    if kind == "train":
        return _train(prepare(case, seed), case)
    if _pairs(case) > (EXACT_RAYS if kind == "raytrace" else EXACT_PAIRS):
        return None
    cfgs = _cfgs(case, seed)
    if kind == "raytrace":
        return _rays(cfgs[0], seed)
    if kind == "two_medium":
        return _two_medium(cfgs[0], seed)
    imgs = [_image(c, seed) for c in cfgs]
    if kind == "multi":
        return imgs
    return torch.cat([i.reshape(-1) for i in imgs]) if kind == "scan" else imgs[0]

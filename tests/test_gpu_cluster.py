"""The clustered stage kernel (stage_cluster.cu) against the direct kernel
(variant 3) and the FP64 kernel on the same points.

Tolerance against FP64, derived: a pair of clusters is interpolated to 5e-7 of
a term at most, and its phases, moments and node terms carry the FP32 rounding
of the direct sum's terms, about 1e-6; incoherent over the clusters, the
relative L2 error of a field stays below 5e-6 plus what the direct kernel has."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2408_06765_gb300 import build, rsi, workloads

pytestmark = pytest.mark.gpu
TOL = 5e-6


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def disk(n, tilt=0.0, **kw):
    return rsi.make_qmc_points(dict({"kind": "disk", "centre": (0.0, 0.0, 0.0), "a": 6.35e-3, "tilt": tilt}, **kw), 3, 0, n)


def rect(n, z, w=0.05, cx=0.0, set_id=1, **kw):
    return rsi.make_qmc_points(dict({"kind": "rect", "centre": (cx, 0.0, z), "wx": w, "wy": w}, **kw), 3, set_id, n)


def grid(nx, nz, z0, z1, half=0.02):
    return rsi.grid_points({"x0": -half, "x1": half, "nx": nx, "z0": z0, "z1": z1, "nz": nz})


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


def fields(kind, k, src, sigma, tgt, **kw):
    return [rsi.propagate_stage(rsi.stage_struct(kind, prec, k, variant=var, **kw), src, sigma, tgt)
            for prec, var in (("fp64", 0), ("fp32c", 3), ("fp32c", 0))]


# (sources, targets): tiles of 128 and 256; ragged last tile, group, root and
# block; grids whose rows are and are not a multiple of the block's strips
PISTON = [
    (lambda: disk(8192), lambda: rect(65536, 0.06)),
    (lambda: disk(9001, 0.17), lambda: rect(60001, 0.06, cx=0.01)),
    (lambda: disk(16385), lambda: grid(257, 129, 0.04, 0.08)),
    (lambda: disk(20011, -0.1), lambda: grid(512, 64, 0.04, 0.09)),
]


@pytest.mark.parametrize("case", range(len(PISTON)))
def test_piston_stage_matches_direct_and_fp64(case):
    src, tgt = (f() for f in PISTON[case])
    exact, direct, clustered = fields(rsi.STAGE_PISTON, 2 * math.pi * 2e6 / 1480.0, src, None, tgt)
    rsi.sync_status()
    assert not torch.equal(clustered, direct)  # the clustered kernel ran
    assert rel(clustered, exact) <= rel(direct, exact) + TOL


@pytest.mark.parametrize("n_src,tgt", [
    (65536, lambda: grid(256, 250, 0.07, 0.11)),
    (70001, lambda: grid(131, 127, 0.05, 0.10)),  # near and far tiles, odd rows
    (262144, lambda: rect(4099, 0.09, set_id=5)),
])
def test_rsi_stage_matches_direct_and_fp64(n_src, tgt):
    src, tgt = rect(n_src, 0.05, w=0.03), tgt()
    k1, k2 = 2 * math.pi * 2e6 / 1480.0, 2 * math.pi * 2e6 / 5900.0
    sigma = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", k1, variant=3), disk(4096), None, src)
    exact, direct, clustered = fields(rsi.STAGE_RSI, k2, src, sigma, tgt)
    rsi.sync_status()
    assert not torch.equal(clustered, direct)
    assert rel(clustered, exact) <= rel(direct, exact) + TOL
    # reversed normals: the exact negation
    neg = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_RSI, "fp32c", k2, normals=rsi.NORMALS_NEG_Z), src, sigma, tgt)
    assert torch.equal(neg, -clustered)


def test_several_frequencies_match_single_stages():
    src, tgt = disk(16384), rect(65536, 0.06)
    ks = [2 * math.pi * f / 1480.0 for f in (1e6, 1.7e6, 2e6)]
    st = rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", ks[0])
    got = rsi.propagate_stage_multi(st, ks, src, None, tgt)
    for f, k in enumerate(ks):
        one = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", k), src, None, tgt)
        assert rel(got[f], one) <= 1e-6  # the same clusters, other splits


@pytest.mark.parametrize("case", ["halton", "curved targets", "too close"])
def test_stages_without_clusters_take_the_direct_kernel(case):
    """Sources in index order, targets off a plane and interfaces a fraction of
    a cluster apart leave no pairs of clusters: the direct kernel's bits."""
    src, z = rect(32768, 0.05), 0.07
    tgt = rect(32768, z, set_id=2)
    if case == "halton":
        src = rect(32768, 0.05, sequence="halton")
    elif case == "curved targets":
        tgt = rsi.make_qmc_points({"kind": "cyl", "centre": (0.0, 0.0, z), "wx": 0.05, "wy": 0.05, "R": 0.1}, 3, 2, 32768)
    else:
        tgt = rect(32768, 0.0501, set_id=2)
    sigma = torch.ones(src.n, dtype=torch.complex128, device="cuda")
    k = 2 * math.pi * 8e6 / 1480.0
    a, b = (rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_RSI, "fp32c", k, variant=v), src, sigma, tgt) for v in (0, 3))
    rsi.sync_status()
    assert torch.equal(a, b)


@pytest.mark.parametrize("case", ["steep", "ragged", "into the slower medium", "near the interface"])
def test_raytrace_matches_direct_and_oracle(case):
    """The clustered ray-tracing sum against the direct one (a given tile) and the FP64 oracle at pixels over the image, by the same
    tolerance: edges of tiles and blocks, rows off the block's strips, rays
    close to the plane (left to the direct sum) and up to 75 degrees."""
    n, nx, nz = {"steep": (16384, 256, 96), "ragged": (9001, 257, 171)}.get(case, (20011, 131, 130))
    cfg = workloads.f2_ray_tracing(n_piston=n, nx=nx, nz=nz)
    g, zi = cfg["grid"], float(cfg["interfaces"][0]["centre"][2])
    if case == "steep":
        g.update({"x0": -0.03, "x1": 0.03})
    elif case == "into the slower medium":
        cfg["media"] = cfg["media"][::-1]
    elif case == "near the interface":
        g.update({"z0": zi + 1e-5, "z1": zi + 0.02})
    clustered, direct = rsi.run_raytrace(cfg), rsi.run_raytrace(cfg, tile=128 if n == 9001 else 256)
    rsi.sync_status()
    assert not torch.equal(clustered, direct)
    assert rel(clustered, direct) <= TOL
    px = np.linspace(0, nx * nz - 1, 64).astype(np.int64)
    want = torch.from_numpy(oracle.raytrace_image(cfg, pixels=px))
    got, ref = (v.reshape(-1).cpu()[torch.from_numpy(px)] for v in (clustered, direct))
    assert rel(got, want) <= rel(ref, want) + TOL

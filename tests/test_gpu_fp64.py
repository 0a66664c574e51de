"""The FP64 stage kernel (stage_fp64.cu) against extended precision on the
same points, where a pair's way changes: lengths from the closest fast pair
(1e-8 m) to the farthest phase (2^18 quarter turns), ragged tiles, amplitudes
of any unit, both normals.

Tolerance, derived: a term is about 16 operations of 2^-48 (6e-14) after a
phase whose path carries 2 roundings of 2^-53 and, in doubles throughout, the
rounding of k r as well: |error| <= sum of |terms| x (1e-13 + k r 2^-51)."""
import math

import numpy as np
import pytest
import torch

from paper_2408_06765_gb300 import build, rsi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def fields(pts, *names):
    return [pts.field(n).cpu().numpy().astype(np.longdouble) for n in names]


@pytest.mark.parametrize("scale,kr", [(1.0, 1000.0), (1.0, 3.9e5), (3e-8, 1.0), (2e3, 50.0), (1.0, 1e-6)])
@pytest.mark.parametrize("n_src,n_tgt,v0", [(1, 1, 1.0), (33, 129, 1e-30), (700, 260, 1e25)])
@pytest.mark.parametrize("kind", ["piston", "plane", "curved"])
def test_terms_match_extended_precision(kind, n_src, n_tgt, v0, scale, kr):
    shape = {"kind": "rect", "centre": (0.0, 0.0, 0.0), "wx": scale, "wy": scale}
    if kind == "curved":
        shape = dict(shape, kind="cyl", R=2.0 * scale)
    src = rsi.make_qmc_points(shape, 1, 0, n_src)
    tgt = rsi.make_qmc_points({"kind": "rect", "centre": (0.1 * scale, 0.0, 0.3 * scale), "wx": scale, "wy": scale}, 1, 1, n_tgt)
    k = kr / scale
    x, y, z, nx, ny, nz, w = fields(src, "X", "Y", "Z", "NX", "NY", "NZ", "W")
    q = [v[:, None] for v in fields(tgt, "X", "Y", "Z")]
    dx, dy, dz = q[0] - x, q[1] - y, q[2] - z
    r = np.sqrt(dx * dx + dy * dy + dz * dz)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    phase = np.exp(1j * (np.longdouble(k) * r))
    if kind == "piston":
        st = rsi.stage_struct(rsi.STAGE_PISTON, "fp64", k, v0)
        got = rsi.propagate_stage(st, src, None, tgt)
        terms = -np.longdouble(v0) * w / (2 * pi * r) * phase
    else:
        rng = np.random.default_rng(n_src)
        sig = (rng.normal(size=n_src) + 1j * rng.normal(size=n_src)) * v0
        normals = rsi.NORMALS_Z if kind == "plane" else rsi.NORMALS_POINTS
        got = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_RSI, "fp64", k, normals=normals), src,
                                  torch.tensor(sig, device="cuda"), tgt)
        nd = dz if kind == "plane" else nx * dx + ny * dy + nz * dz
        terms = -w * sig.astype(np.clongdouble) / (2 * pi) * (1j * np.longdouble(k) - 1 / r) * phase * nd / r / r
        # the size of a term before the obliquity, whose own rounding is relative to |d|
        phase = w * np.abs(sig) / (2 * pi) * np.abs(1j * np.longdouble(k) - 1 / r) / r
    rsi.sync_status()
    size = np.abs(terms) if kind == "piston" else phase
    bound = (size * (1e-13 + np.longdouble(k) * r * 2.0 ** -51)).sum(1)
    assert np.all(np.abs(got.cpu().numpy() - terms.sum(1)) <= bound)


def test_short_paths_keep_their_phase():
    """The phase of single pairs of 0.5 to 10 radians.  What is left of a quarter
    turn times the distance's correction is a float below 0.6 x 2^-22, rounded
    twice: 2^-48 quarter turns at most, 3.2e-15 rad rms each; sine, cosine and
    their products add six roundings of 2^-48, 2e-15 rms each."""
    src = rsi.make_qmc_points({"kind": "rect", "centre": (0.0, 0.0, 0.0), "wx": 1e-3, "wy": 1e-3}, 1, 0, 1)
    tgt = rsi.make_qmc_points({"kind": "rect", "centre": (0.0, 0.0, 0.05), "wx": 2.0, "wy": 2.0}, 1, 1, 4096)
    k = 7.0
    got = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp64", k), src, None, tgt).cpu().numpy()
    rsi.sync_status()
    p = fields(src, "X", "Y", "Z")
    r = np.sqrt(sum((a - b) ** 2 for a, b in zip(fields(tgt, "X", "Y", "Z"), p)))
    # the field's sign is -1: the angle between it and -e^{ikr}
    c, s = np.cos(np.longdouble(k) * r), np.sin(np.longdouble(k) * r)
    re, im = got.real.astype(np.longdouble), got.imag.astype(np.longdouble)
    off = (im * c - re * s) / np.sqrt(re * re + im * im)
    assert float(np.sqrt(np.mean(off * off))) <= 7e-15


@pytest.mark.parametrize("kind", ["piston", "plane", "curved"])
def test_variant_1_keeps_doubles(kind):
    """Every operation in doubles: some 12 roundings of 2^-53 a term and, of its
    phase, that of k r and of the distance."""
    shape = {"kind": "cyl" if kind == "curved" else "rect", "centre": (0.0, 0.0, 0.0), "wx": 0.03, "wy": 0.03, "R": 0.1}
    src = rsi.make_qmc_points(shape, 1, 0, 700)
    tgt = rsi.make_qmc_points({"kind": "rect", "centre": (0.0, 0.0, 0.05), "wx": 0.03, "wy": 0.03}, 1, 1, 260)
    k = 8000.0
    x, y, z, nx, ny, nz, w = fields(src, "X", "Y", "Z", "NX", "NY", "NZ", "W")
    q = [v[:, None] for v in fields(tgt, "X", "Y", "Z")]
    dx, dy, dz = q[0] - x, q[1] - y, q[2] - z
    r = np.sqrt(dx * dx + dy * dy + dz * dz)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    phase, sigma, normals = np.exp(1j * (np.longdouble(k) * r)), None, rsi.NORMALS_Z
    terms = -w / (2 * pi * r) * phase
    if kind != "piston":
        sigma = torch.full((src.n,), 0.6 - 0.8j, dtype=torch.complex128, device="cuda")
        normals = rsi.NORMALS_Z if kind == "plane" else rsi.NORMALS_POINTS
        nd = dz if kind == "plane" else nx * dx + ny * dy + nz * dz
        s = np.clongdouble(complex(0.6, -0.8))
        terms = -w * s / (2 * pi) * (1j * np.longdouble(k) - 1 / r) * phase * nd / r / r
    what = rsi.STAGE_PISTON if kind == "piston" else rsi.STAGE_RSI
    got, auto = (rsi.propagate_stage(rsi.stage_struct(what, "fp64", k, normals=normals, variant=v), src, sigma, tgt)
                 for v in (1, 0))
    rsi.sync_status()
    assert not torch.equal(got, auto)
    size = np.abs(terms) if kind == "piston" else w / (2 * pi) * np.abs(1j * np.longdouble(k) - 1 / r) / r
    bound = (size * (12 * 2.0 ** -53 + np.longdouble(k) * r * 2.0 ** -52)).sum(1)
    assert np.all(np.abs(got.cpu().numpy() - terms.sum(1)) <= bound)

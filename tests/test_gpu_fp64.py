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

"""The clustered sums (stage_cluster.cu, raytrace.cu) on target sets and
amplitudes that the other tests do not have.

Tolerance against FP64 as in test_gpu_cluster.py: 5e-6 beyond the direct
sum's own error, here with the worst value bounded as well."""
import ctypes
import math

import pytest
import torch

from fieldcheck import assert_close, rel_l2
from paper_2408_06765_gb300 import build, rsi, workloads

pytestmark = pytest.mark.gpu
TOL = 5e-6
K_WATER, K_STEEL = (2 * math.pi * 2e6 / c for c in (1480.0, 5900.0))


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()


def disk(n, tilt=0.0):
    return rsi.make_qmc_points({"kind": "disk", "centre": (0.0, 0.0, 0.0), "a": 6.35e-3, "tilt": tilt}, 3, 0, n)


def interface(n, z=0.05, w=0.03):
    return rsi.make_qmc_points({"kind": "rect", "centre": (0.0, 0.0, z), "wx": w, "wy": w}, 3, 1, n)


def image(nx, nz, z0, z1, half=0.02):
    return rsi.grid_points({"x0": -half, "x1": half, "nx": nx, "z0": z0, "z1": z1, "nz": nz})


def points(x, y, z):
    """A target set of a caller's own coordinates (float64 tensors), in the order given."""
    pts = rsi.Points(x.numel())
    pts.buf.zero_()
    for name, v in (("X", x), ("Y", y), ("Z", z)):
        set_coordinate(pts, name, slice(None), v.reshape(-1).cuda())
    return pts


def set_coordinate(pts, name, at, v):
    hi = torch.as_tensor(v, dtype=torch.float64).to(torch.float32)
    pts.field(name)[at] = v
    pts.field(name + "H")[at] = hi.cuda()
    pts.field(name + "L")[at] = (torch.as_tensor(v, dtype=torch.float64) - hi.double()).float().cuda()


def volume(nx, ny, nz, step, z0, slow=("z", "y")):
    """A box of targets, x fastest, then y and z, or z and y."""
    ax = {"x": (torch.arange(nx, dtype=torch.float64) - nx / 2) * step,
          "y": (torch.arange(ny, dtype=torch.float64) - ny / 2) * step,
          "z": torch.arange(nz, dtype=torch.float64) * step + z0}
    c = dict(zip(slow + ("x",), torch.meshgrid(*(ax[a] for a in slow + ("x",)), indexing="ij")))
    return points(c["x"], c["y"], c["z"])


def stage_fields(kind, k, src, sigma, tgt):
    return [rsi.propagate_stage(rsi.stage_struct(kind, prec, k, variant=var), src, sigma, tgt)
            for prec, var in (("fp64", 0), ("fp32c", 3), ("fp32c", 0))]


# Targets in rows of which a block of 1024 spans two planes and a quarter of it
# one: strips of 32 slices of a volume, two rows of y each; images 48 rows high
# one behind the other in y, 8 and 1 mm apart; all against a tilted piston and
# an interface below which they lie.
SETS = {
    "volume": lambda: volume(48, 32, 64, 0.5e-3, 0.06),
    "images": lambda: volume(128, 8, 48, 0.25e-3, 0.07, slow=("y", "z")),
    "thin stack": lambda: volume(256, 5, 48, 0.1e-3, 0.08, slow=("y", "z")),
}


@pytest.mark.parametrize("kind", ["piston", "interface"])
@pytest.mark.parametrize("name", list(SETS))
def test_targets_off_a_plane_match_fp64(name, kind):
    tgt = SETS[name]()
    if kind == "piston":
        exact, direct, got = stage_fields(rsi.STAGE_PISTON, K_WATER, disk(16384, 0.1), None, tgt)
    else:
        src = interface(65536)
        sigma = rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", K_WATER, variant=3), disk(4096), None, src)
        exact, direct, got = stage_fields(rsi.STAGE_RSI, K_STEEL, src, sigma, tgt)
    rsi.sync_status()
    own = rel_l2(direct.cpu(), exact.cpu())
    assert_close(got.cpu(), exact.cpu(), own + TOL, name)


@pytest.mark.parametrize("first,count", [(37, 128 * 300), (300, 40001), (128 * 64, 128 * 256)])
def test_slices_of_an_image_match_fp64(first, count):
    """A share of an image's slots, from within a row or in ragged numbers."""
    tgt = rsi.points_slice(image(128, 512, 0.05, 0.09), first, count)
    exact, direct, got = stage_fields(rsi.STAGE_PISTON, K_WATER, disk(20011, 0.1), None, tgt)
    rsi.sync_status()
    assert not torch.equal(got, direct)  # the clustered kernel ran
    assert_close(got.cpu(), exact.cpu(), rel_l2(direct.cpu(), exact.cpu()) + TOL)


@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf])
@pytest.mark.parametrize("coordinate", ["X", "Y", "Z"])
@pytest.mark.parametrize("kind", ["piston", "raytrace"])
def test_a_target_that_is_no_number_is_reported(kind, coordinate, value):
    """... and leaves every other target as it was."""
    tgt, at = image(256, 256, 0.06, 0.10), 256 * 100 + 37
    if kind == "piston":
        src = disk(16384)
        run = lambda: rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", K_WATER), src, None, tgt)
    else:
        cfg = workloads.f2_ray_tracing(n_piston=16384, nx=256, nz=256)
        src, tgt = disk(16384), rsi.grid_points(cfg["grid"])
        run = lambda: rsi.raytrace_field(rsi.raytrace_struct(cfg), src, tgt)
    want = run()
    rsi.sync_status()
    set_coordinate(tgt, coordinate, at, value)
    got = run()
    with pytest.raises(rsi.RSIError):
        rsi.sync_status()
    assert not torch.isfinite(torch.view_as_real(got[at])).all()
    got[at] = want[at]
    assert rel_l2(got.cpu(), want.cpu()) <= TOL


@pytest.mark.parametrize("kind", ["piston", "interface", "raytrace"])
@pytest.mark.parametrize("power", [-80, -60, 60, 80])
def test_fields_are_linear_in_the_amplitude(kind, power):
    """A power of two of the velocity or density is one of the field.  Every
    product and sum of the kernel keeps its bits under it as long as nothing
    leaves the range of FP32; the smallest moments' parts do at 2^-80, by
    2^-149 / 2^-110 of the largest."""
    s = 2.0 ** power

    def run(s):
        if kind == "piston":
            st = rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", K_WATER, s)
            return rsi.propagate_stage(st, disk(16384), None, image(256, 256, 0.06, 0.10))
        if kind == "interface":
            src = interface(65536)
            sigma = torch.full((src.n,), s, dtype=torch.complex128, device="cuda")
            return rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_RSI, "fp32c", K_STEEL), src, sigma, image(256, 192, 0.07, 0.11))
        cfg = workloads.f2_ray_tracing(n_piston=16384, nx=256, nz=256)
        cfg["v0"] = s
        return rsi.raytrace_field(rsi.raytrace_struct(cfg), disk(16384), rsi.grid_points(cfg["grid"]))

    one, got = run(1.0), run(s)
    rsi.sync_status()
    assert float(torch.linalg.vector_norm(got)) > 0.0
    assert_close((got / s).cpu(), one.cpu(), 1e-7)


@pytest.mark.parametrize("kind", ["piston", "several frequencies", "raytrace"])
def test_a_workspace_for_the_direct_sum_gets_the_direct_sum(kind):
    """A scratch buffer of the direct sum's size, and nothing smaller."""
    lib, src, tgt = rsi.load(), disk(16384), image(256, 256, 0.06, 0.10)
    out = torch.empty((3, tgt.n), dtype=torch.complex128, device="cuda")
    ks = (ctypes.c_double * 3)(K_WATER, 1.3 * K_WATER, 1.7 * K_WATER)
    cfg = workloads.f2_ray_tracing(n_piston=16384, nx=256, nz=256)
    if kind == "raytrace":
        tgt = rsi.grid_points(cfg["grid"])
    stream = rsi._stream()

    def call(ask, nbytes=None):
        """The size asked for, or the call with a buffer of so many bytes."""
        if kind == "raytrace":
            st = rsi.raytrace_struct(cfg, tile=256 if ask else 0)
            args = (src.ptr(), src.n, tgt.ptr(), tgt.n, rsi._ptr(out))
            size, run = lib.rsi_raytrace_workspace_bytes(ctypes.byref(st), src.n, tgt.n), lib.rsi_raytrace_field
        else:
            st = rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", K_WATER, variant=3 if ask else 0)
            args = (src.ptr(), src.n, None, tgt.ptr(), tgt.n, rsi._ptr(out))
            if kind == "piston":
                size, run = lib.rsi_stage_workspace_bytes(ctypes.byref(st), src.n, tgt.n), lib.rsi_propagate_stage
            else:
                size = lib.rsi_stage_multi_workspace_bytes(ctypes.byref(st), 3, ks, src.n, tgt.n)
                run, args = lib.rsi_propagate_stage_multi, (3, ks) + args
        if nbytes is None:
            return size
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        out.fill_(0)
        rc = run(ctypes.byref(st), *args, rsi._ptr(ws), nbytes, stream)
        return rc, out.clone()

    small, large = call(True), call(False)
    assert small < large
    rc, want = call(True, small)
    assert rc == 0
    for nbytes in (small, large - 1):
        rc, got = call(False, nbytes)
        assert rc == 0 and torch.equal(got, want)
    rc, got = call(False, large)
    assert rc == 0 and not torch.equal(got, want)
    assert call(False, small - 1)[0] == -5  # RSI_E_NOMEM
    rsi.sync_status()


@pytest.mark.parametrize("n,nx,nz", [(19000, 129, 127), (9300, 256, 128)])
def test_short_ray_sums_take_the_direct_kernel(n, nx, nz):
    """3e8 rays: the clustered sum took 1.1 to 1.3 times as long."""
    cfg = workloads.f2_ray_tracing(n_piston=n, nx=nx, nz=nz)
    got, direct = rsi.run_raytrace(cfg), rsi.run_raytrace(cfg, tile=128 if n < 16384 else 256)
    rsi.sync_status()
    assert torch.equal(got, direct)


def test_a_short_sum_close_to_its_interface_takes_the_direct_kernel():
    """1e9 pairs, most clusters too close: the clustered sum took 1.14 times as long."""
    k, src, tgt = 2 * math.pi * 5e6 / 5900.0, interface(61100), image(128, 128, 0.0505, 0.09)
    sigma = torch.ones(src.n, dtype=torch.complex128, device="cuda")
    got, direct = (rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_RSI, "fp32c", k, variant=v), src, sigma, tgt)
                   for v in (0, 3))
    rsi.sync_status()
    assert torch.equal(got, direct)


@pytest.mark.parametrize("variant", [1, 2, 3])
def test_a_variant_asks_for_the_direct_sums_of_several_frequencies(variant):
    cfgs = []
    for f in (2e6, 3e6):
        cfg = workloads.c2_full_image(f)
        cfg["piston"]["n"], cfg["interfaces"][0]["n"] = 16384, 65536
        cfg["grid"].update({"nx": 256, "nz": 192})
        cfgs.append(cfg)
    got = rsi.run_chain_multi(cfgs, stage_opts={"variant": variant})
    want = rsi.run_chain_multi(cfgs, stage_opts={"tile": 256})
    clustered = rsi.run_chain_multi(cfgs)
    rsi.sync_status()
    for a, b, c in zip(got, want, clustered):
        assert torch.equal(a, b) and not torch.equal(a, c)


@pytest.mark.parametrize("kind,freqs", [
    ("piston", (1e6, 1.7e6, 2e6)), ("interface", (1e6, 1.7e6)), ("interface", (1e6, 1.7e6, 2e6)),
    ("interface", (1e6, 1.3e6, 1.7e6, 1.9e6)),
])
def test_several_frequencies_take_clusters_and_match_fp64(kind, freqs):
    """Each frequency with a density of its own; three of them with and four
    without one that is twice another."""
    ks = [2 * math.pi * f / (1480.0 if kind == "piston" else 5900.0) for f in freqs]
    if kind == "piston":
        src, sigma, tgt, what = disk(16384), None, image(256, 256, 0.06, 0.10), rsi.STAGE_PISTON
    else:
        src, tgt, what = interface(65536), image(256, 192, 0.07, 0.11), rsi.STAGE_RSI
        sigma = torch.stack([rsi.propagate_stage(rsi.stage_struct(rsi.STAGE_PISTON, "fp32c", 2 * math.pi * f / 1480.0, variant=3),
                                                 disk(4096), None, src) for f in freqs])
    got, direct = (rsi.propagate_stage_multi(rsi.stage_struct(what, "fp32c", ks[0], variant=v), ks, src, sigma, tgt)
                   for v in (0, 3))
    rsi.sync_status()
    for f, k in enumerate(ks):
        exact = rsi.propagate_stage(rsi.stage_struct(what, "fp64", k), src, None if sigma is None else sigma[f], tgt)
        assert not torch.equal(got[f], direct[f])
        assert_close(got[f].cpu(), exact.cpu(), rel_l2(direct[f].cpu(), exact.cpu()) + TOL, f"{freqs[f]:g} Hz")

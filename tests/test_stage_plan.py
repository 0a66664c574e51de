"""Which sums are offered clusters, and what scratch they ask for beside the
direct sum's, from the library's own plans (no GPU needed)."""
import ctypes

import pytest

from paper_2408_06765_gb300 import build, rsi, workloads

GIB = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()


def extra(n_src, n_tgt, kind=rsi.STAGE_PISTON):
    auto, direct = (rsi.workspace_bytes(rsi.stage_struct(kind, "fp32c", 1e3, variant=v), n_src, n_tgt) for v in (0, 3))
    return auto - direct


@pytest.mark.parametrize("n_src,n_tgt", [(1 << 27, 1 << 27), (8192, 1 << 31), (1 << 31, 8192)])
def test_tables_beyond_an_eighth_of_the_memory_are_not_asked_for(n_src, n_tgt):
    assert extra(n_src, n_tgt) == 0


@pytest.mark.parametrize("n_src,n_tgt", [(8192, 65536), (16384, 65536), (1 << 20, 1 << 20), (1 << 26, 1 << 26)])
def test_long_piston_sums_are_offered_clusters(n_src, n_tgt):
    assert 0 < extra(n_src, n_tgt) <= 32 * GIB


@pytest.mark.parametrize("n,nx,nz,offered", [(19000, 129, 127, False), (9300, 256, 128, False), (20011, 131, 130, True),
                                             (65536, 512, 512, True), (131072, 64, 64, False)])
def test_ray_sums_are_offered_clusters_where_they_pay(n, nx, nz, offered):
    cfg = workloads.f2_ray_tracing(n_piston=n, nx=nx, nz=nz)
    auto, direct = (rsi.load().rsi_raytrace_workspace_bytes(ctypes.byref(rsi.raytrace_struct(cfg, newton=k)), n, nx * nz)
                    for k in (0, 1))
    assert (auto > direct) == offered

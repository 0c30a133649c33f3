"""The C-ABI library loads on a machine without a GPU and exports every entry
point that include/stokes.h declares; argument errors are reported without
touching the device."""
import ctypes
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2509_19061_gb300 import build
    path = build.build()
    return ctypes.CDLL(path)


def declared_symbols():
    with open(os.path.join(ROOT, "include", "stokes.h")) as f:
        text = f.read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(stokes_[a-z_0-9]+)\s*\(", text)))


def test_header_declares_the_boundary():
    syms = declared_symbols()
    for name in ("stokes_create", "stokes_get_layout", "stokes_set_viscosity", "stokes_set_rhs",
                 "stokes_apply_operator", "stokes_smooth", "stokes_residual_energy_norm", "stokes_vcycle",
                 "stokes_destroy", "stokes_strerror"):
        assert name in syms


def test_library_exports_every_declared_symbol(lib):
    missing = [s for s in declared_symbols() if not hasattr(lib, s)]
    assert not missing, missing


def test_binding_covers_every_declared_symbol():
    from paper_2509_19061_gb300 import api
    assert set(declared_symbols()) <= set(api.exported_symbols())


def test_argument_errors_without_device(lib):
    from paper_2509_19061_gb300 import api
    out = ctypes.c_void_p(123)
    f = api._lib()
    assert f.stokes_create(1, 8, 1.0, 1.0, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert out.value is None
    assert f.stokes_create(8, 8, 0.0, 1.0, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert f.stokes_create(8, 8, 1.0, 1.0, 7, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert f.stokes_create((1 << 18) + 1, 8, 1.0, 1.0, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert f.stokes_create(8, (1 << 18) + 1, 1.0, 1.0, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert f.stokes_get_layout(None, 0, None, None, None, None) == api.STOKES_ERR_ARG
    assert f.stokes_smooth(None, None, None, None, None) == api.STOKES_ERR_ARG
    assert f.stokes_destroy(None) == api.STOKES_OK
    assert f.stokes_strerror(api.STOKES_ERR_DIVERGED).decode().startswith("diverged")
    assert f.stokes_set_option(None, api.STOKES_OPT_PAIRED, 1) == api.STOKES_ERR_ARG
    for bad in [(0, 8, 8, 8, 1, 0, 1, 1), (8, 8, 8, 8, -1, 0, 1, 1), (8, 8, 8, 8, 1, 2, 1, 1),
                (8, 8, 8, 8, 1, 0, 1, 3), (8, 8, 0, 8, 1, 0, 1, 1)]:
        assert f.stokes_tile_kernel_plan(*bad, None, None, None) == api.STOKES_ERR_ARG, bad


def test_product_path_has_no_oracle_dependency():
    """The package never imports the oracle or falls back to CPU code."""
    pkg = os.path.join(ROOT, "paper_2509_19061_gb300")
    for dirpath, _, files in os.walk(pkg):
        for fn in files:
            if fn.endswith((".py", ".cu", ".h", ".cuh")):
                with open(os.path.join(dirpath, fn)) as f:
                    src = f.read()
                assert "import oracle" not in src and "from oracle" not in src, fn
                assert "stokes_oracle" not in src, fn


def test_batch_argument_errors_without_device(lib):
    from paper_2509_19061_gb300 import api
    f = api._lib()
    out = ctypes.c_void_p(123)
    n2 = (ctypes.c_int * 2)(32, 1)
    l2 = (ctypes.c_double * 2)(1.0, 1.0)
    assert f.stokes_batch_create(2, n2, n2, l2, l2, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert out.value is None
    assert f.stokes_batch_create(0, n2, n2, l2, l2, 1, None, ctypes.byref(out)) == api.STOKES_ERR_ARG
    assert f.stokes_batch_get_layout(None, 0, None, None, None) == api.STOKES_ERR_ARG
    assert f.stokes_batch_smooth(None, None, None, None, None) == api.STOKES_ERR_ARG
    assert f.stokes_batch_solve(None, None, None, None, None, None, None, None) == api.STOKES_ERR_ARG
    assert f.stokes_batch_destroy(None) == api.STOKES_OK


def test_batched_workload_recipe():
    """Sides are multiples of 64 between 64 and 1024 (so that halving reaches
    a coarsest level of at most 16 x 16 cells), contrasts in [1e2, 1e6],
    sinkers inside the box; the table is a pure function of the seed."""
    from paper_2509_19061_gb300 import inputs
    a = inputs.batch_specs(seed=5, count=256)
    assert a == inputs.batch_specs(seed=5, count=256)
    ns = [s.n for s in a]
    assert all(n % 64 == 0 and 64 <= n <= 1024 for n in ns)
    assert len(set(ns)) >= 12
    for n in ns:
        m = n
        while m % 2 == 0 and m > 16:
            m //= 2
        assert 2 * m * (m - 1) <= 1024
    assert all(1e2 <= s.contrast <= 1e6 for s in a)
    assert all(s.radius + 0.3 > 0 and 0.05 <= s.radius <= 0.2 and 0.3 <= s.cx <= 0.7 for s in a)
    cells = np.array([n * n for n in ns], dtype=np.float64)
    assert 1.0e5 < cells.mean() < 3.0e5


@pytest.mark.parametrize("dtype,nx,ny", [("f64", 64, 64), ("f64", 2, 2), ("f64", 250, 18), ("f32", 128, 128),
                                         ("f32", 33, 31), ("f32", 256, 9), ("f32", 31, 500)])
def test_small_grids_fit_the_clusters_that_a_device_runs(lib, dtype, nx, ny):
    """A schedule that one cluster of CTAs runs is planned for the largest cluster
    that the device has room for, down to one CTA, and goes back to the tiles
    where that does not hold the grid; no device is read."""
    from paper_2509_19061_gb300 import api
    ras = api.smooth_params("ras", sweeps=10, tile=(16, 16), k=4, overlap=3)
    was = None
    for most in (1, 2, 4, 8, 16):
        plan = api.stokes_smooth_plan(nx, ny, ras, dtype, max_cluster=most)
        if plan["path"] == "cluster":
            assert 1 <= plan["cluster"] <= most and plan["passes"] == 1
            assert was in (None, "tiles", "cluster")
        else:
            assert plan["path"] == "tiles" and was != "cluster"
        was = plan["path"]
    assert was == "cluster"


def test_smooth_plan_without_device(lib):
    """What stokes_smooth runs, by variant, size, dtype and option."""
    from paper_2509_19061_gb300 import api

    def plan(n, dtype="f32", m=None, use_tma=True, pair_mode=1, **kw):
        return api.stokes_smooth_plan(n, m or n, api.smooth_params(**kw), dtype, use_tma, pair_mode, 16)

    exact = dict(variant="ras", sweeps=20, tile=(32, 32), k=4, overlap=3)
    assert plan(8192, **exact) == dict(path="stream", passes=3, tile=(0, 0), k=0, overlap=0, cluster=0)
    assert plan(1024, "f64", **exact)["path"] == "stream" and plan(1024, "f64", **exact)["passes"] == 5
    assert plan(8192, pair_mode=2, **exact) == dict(path="tiles", passes=5, tile=(32, 32), k=4, overlap=3, cluster=0)
    assert plan(8192, use_tma=False, **exact)["path"] == "tiles"
    mid = plan(512, **exact)
    assert mid["path"] == "tiles" and mid["tile"][0] == 64 - 2 * mid["k"] and mid["overlap"] == mid["k"] - 1
    assert plan(128, **exact)["path"] == "cluster"
    assert plan(8192, **dict(exact, overlap=0))["tile"] == (32, 32)
    assert plan(2000, variant="rbgs", sweeps=5) == dict(path="stream", passes=3, tile=(0, 0), k=0, overlap=0, cluster=0)
    assert plan(2000, variant="rbgs", sweeps=1)["path"] == "passes"
    assert plan(2000, variant="jacobi", sweeps=7) == dict(path="passes", passes=7, tile=(0, 0), k=0, overlap=0, cluster=0)
    assert plan(2000, variant="blocked", sweeps=7, tile=(24, 16))["tile"] == (24, 16)
    assert plan(64, **dict(exact, sweeps=0))["passes"] == 0
    for bad in (dict(variant="mixed"), dict(exact, k=0, overlap=0), dict(exact, pair_mode=3), dict(exact, dtype=7)):
        kw = dict(bad)
        with pytest.raises(api.StokesError):
            if kw.pop("dtype", None) == 7:
                st = api._lib().stokes_smooth_plan(8, 8, 7, ctypes.byref(api.smooth_params(**kw)), 1, 1, 16,
                                                   ctypes.byref(api.stokes_smooth_plan_info()))
                raise api.StokesError(st, "dtype")
            plan(64, **kw)


def test_narrow_grids_keep_their_tiles(lib):
    """A row-streaming strip sweeps its full width however few columns the grid
    has: RAS and RBGS on narrow grids run on tiles, fused Jacobi streams."""
    from paper_2509_19061_gb300 import api

    def path(nx, ny, dtype, **kw):
        return api.stokes_smooth_plan(nx, ny, api.smooth_params(**kw), dtype, max_cluster=16)["path"]

    exact = dict(variant="ras", sweeps=8, tile=(32, 32), k=4, overlap=3)
    for dtype, nx in (("f32", 20), ("f64", 32)):
        assert path(nx - 1, 200000, dtype, **exact) == "tiles" and path(nx, 200000, dtype, **exact) == "stream"
        assert path(3, 250000, dtype, variant="fused", sweeps=8) == "stream"
        assert path(250000, 3, dtype, **exact) == "stream"
    assert path(47, 200000, "f32", variant="rbgs", sweeps=6) == "passes"
    assert path(48, 200000, "f32", variant="rbgs", sweeps=6) == "stream"


def test_one_wave_of_given_tiles_stays(lib):
    """Middle FP32 grids whose given tiles run the sweeps in one pass of one wave
    keep them; more sweeps, more tiles or wider windows take chosen ones."""
    from paper_2509_19061_gb300 import api

    def tile(n, sweeps, tile=(32, 32), k=4, overlap=3):
        plan = api.stokes_smooth_plan(n, n, api.smooth_params("ras", sweeps, tile, k, overlap), "f32", max_cluster=16)
        assert plan["path"] == "tiles"
        return plan["tile"]

    assert tile(200, 4) == tile(330, 3) == (32, 32)
    for other in (tile(200, 5), tile(400, 4), tile(200, 4, (56, 32)), tile(200, 8, (30, 30), 8, 7)):
        assert other not in ((32, 32), (30, 30))

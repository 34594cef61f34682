"""The planner of the two-level search, on the host: what it has to leave to the
one-level search."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    """plan(n, epochs, span, n_min, tph, mean_weight, **grid): None (one level) or the two-level plan's sizes."""
    from paper_2509_26279_gb300 import _build
    _build.build()  # before the library is loaded
    from paper_2509_26279_gb300 import sas
    so = str(tmp_path_factory.mktemp("plan") / "plan.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-shared", "-o", so,
                    os.path.join(ROOT, "tests", "native", "plan_windows.cu"), _build.LIB, "-Xlinker",
                    "-rpath=" + _build.OUT_DIR], check=True)
    lib = ctypes.CDLL(so)
    lib.plan_windows_for_test.argtypes = [ctypes.POINTER(sas.sas_grid_desc), ctypes.c_uint64, ctypes.c_uint32, ctypes.c_int64,
                                          ctypes.c_int64, ctypes.c_uint32, ctypes.c_double, ctypes.POINTER(ctypes.c_int64)]
    names = ("gx", "gy", "win", "cell", "units", "rows", "spatial", "list_cap", "counter_bits", "step_x")

    def run(n, epochs, span, n_min, tph=3600, mean_weight=0.0, **grid):
        out = (ctypes.c_int64 * len(names))()
        rc = lib.plan_windows_for_test(ctypes.byref(sas.sas_grid_desc(**grid)), n, epochs, span, tph, n_min, mean_weight, out)
        assert rc >= 0
        return dict(zip(names, out)) if rc else None
    return run


def _grid(nvx=111, nvy=111, dv=364, nbx=1024, nby=2048, bin=2000, **kw):
    g = dict(vx0=-(nvx // 2) * dv, vy0=-(nvy // 2) * dv, dvx=dv, dvy=dv, nvx=nvx, nvy=nvy, x_min=0, y_min=0, nbx=nbx, nby=nby,
             bin=bin, speed_min=0, speed_max=0)
    g.update(kw)
    return g


def test_ordinary_field_is_searched_in_two_levels(plan):
    p = plan(320_000, 100, 14_400, 25, **_grid())
    assert p and p["units"] < 1 << 32


@pytest.mark.parametrize("n", [10**6, 10**8])
def test_more_than_32_bits_of_units(plan, n):
    """134,000 x 134,000 bins and 16 million velocities are inside the library's limits; the units of a level 1 of that
    size do not fit the 32 bits that its kernel numbers them with."""
    p = plan(n, 100, 14_400, 25, **_grid(4001, 4001, 364, 134_000, 134_000))
    assert p is None or p["units"] < 1 << 32


@pytest.mark.parametrize("dv,nv,span", [(3 * 10**8, 14, 6), (3 * 10**8, 14, 20), (5 * 10**8, 8, 20)])
def test_group_steps_beyond_32_bits(plan, dv, nv, span):
    """Steps of some 10^8 mpx/h are legal over a few milliseconds; a group's step of eight of them is not an int32."""
    p = plan(5_000_000, 100, span, 60, tph=3_600_000,
             **_grid(nv, nv, dv, 4096, 4096, vx0=-(nv // 2) * dv + 1000, vy0=-(nv // 2) * dv + 1000))
    assert p is None or p["step_x"] == p["gx"] * dv


def test_centre_velocity_times_time_beyond_64_bits(plan):
    """Twice a centre velocity of 2^31 mpx/h over 2^32 ticks is 2^64; the same lattice over fewer ticks is planned."""
    grid = _grid(75, 83, 3, 1024, 2048, 4000, vx0=2_100_000_000, vy0=2_100_000_000)
    assert plan(2_000_000, 60, 1 << 30, 20, tph=1 << 38, **grid)
    p = plan(2_000_000, 60, (1 << 32) - 1, 20, tph=1 << 40, **grid)
    assert p is None


@pytest.mark.parametrize("lam,n_min", [(400, 25), (540, 64), (812, 90), (812, 128)])
def test_noise_that_fills_every_window(plan, lam, n_min):
    """lam detections per window of 10.6 px on average, far above the threshold: every window would be kept."""
    n = int(lam / 10.6**2 * 2048 * 4096)
    assert plan(n, 255, 14_400, n_min, **_grid()) is None

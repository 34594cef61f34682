"""The two-level window search (the default for large searches) against the
one-level kernel, which a caller's tile sizes select, byte for byte: candidate
records, ids and pair counts, over lattices, domains, epochs and thresholds at
the edges of what the two-level search takes.  The oracle judges one of them."""
import numpy as np
import pytest

import oracle
from paper_2509_26279_gb300 import workloads as W
from tests import cases

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2509_26279_gb300 import sas  # noqa: E402
from tests.test_gpu_parity import assert_same  # noqa: E402


def _field(seed, width=1021, height=1777, epochs=60, noise=700, movers=40, span=4.0):
    r = W.FieldRecipe(width, height, epochs, span, noise, movers, (0.5, 15.0), (0.9, 0.4))
    return W.make_catalog(r, seed)


def _grid(width=1021, height=1777, nvx=75, nvy=83, dvx=364, dvy=364, bin_mpx=2000, x_min=0, y_min=0, **kw):
    return W.GridSpec(vx0=-(nvx // 2) * dvx, vy0=-(nvy // 2) * dvy, dvx=dvx, dvy=dvy, nvx=nvx, nvy=nvy, x_min=x_min,
                      y_min=y_min, nbx=-(-width * 1000 // bin_mpx), nby=-(-height * 1000 // bin_mpx), bin=bin_mpx, **kw)


def _both(cat, grid, n_min, **kw):
    """(default search, one-level search) as bytes, and their infos."""
    out = []
    for tiles in (dict(), dict(tile_kx=8, tile_ky=8)):
        o = sas.make_opts(**tiles)
        for k, v in kw.items():
            setattr(o, k, v)
        res = sas.stack_catalog(sas.Grid(grid), cat, n_min, opts=o)
        c, ids = res.candidates()
        out.append((c.tobytes(), ids.tobytes(), len(c), res.info()))
    return out


def _check(cat, grid, n_min, **kw):
    two, one = _both(cat, grid, n_min, **kw)
    assert two[2] == one[2] and two[0] == one[0] and two[1] == one[1]
    assert two[3]["n_pairs"] == one[3]["n_pairs"] and two[3]["t0"] == one[3]["t0"]
    return two, one


def _shuffled_times(cat):
    """Epoch times out of order, the earliest in the middle, epochs 0 and 7 without detections."""
    t = np.roll(cat.t, 23) + 12345
    keep = (cat.epoch != 0) & (cat.epoch != 7)
    return cases.catalog(cat.x[keep], cat.y[keep], cat.epoch[keep], t, cat.ticks_per_hour)


GRIDS = [
    dict(),
    dict(dvx=-364, dvy=200),                       # one axis backwards, unequal steps: unequal groups
    dict(nvx=73, nvy=1, dvx=364, dvy=0),            # a single lattice row
    dict(nvx=9, nvy=300, dvx=364, dvy=120),
    dict(bin_mpx=2501, x_min=-31000, y_min=17001),  # a domain that is not the field
    dict(speed_min=3000, speed_max=12000),
]


@pytest.mark.parametrize("grid", GRIDS)
def test_lattices_and_domains(grid):
    cat = _field(1)
    two, one = _check(cat, _grid(**grid), 15)
    assert two[2] > 0
    if grid.get("nvy", 83) > 1:
        assert two[3]["n_emitted"] != one[3]["n_emitted"]   # windows, not super-bins: the two-level search ran


@pytest.mark.parametrize("a,b", [(0, 17), (5, 3000), (2100, 75 * 83), (75 * 40, 75 * 41), (75 * 83 - 1, 75 * 83)])
def test_lattice_ranges(a, b):
    _check(_field(2), _grid(), 14, v_begin=a, v_end=b)


@pytest.mark.parametrize("n_min", [5, 7, 8, 9, 16, 40])
def test_thresholds(n_min):
    """Both packings of the window sums (n_min under and over 8) and cells with more than 15 detections."""
    two, _ = _check(_field(3, noise=150, movers=60), _grid(nvx=111, nvy=111), n_min)
    assert two[2] > 0


@pytest.mark.parametrize("epochs,n_min", [(11, 8), (128, 30), (150, 128), (255, 60), (256, 60)])
def test_epoch_counts(epochs, n_min):
    """Few epochs, bucket rows shared by many, the last count that the two-level search takes and the first that it does not."""
    cat = _field(4, epochs=epochs, noise=60000 // epochs, movers=30)
    _check(cat, _grid(), n_min)


def test_times_out_of_order_and_empty_epochs():
    two, _ = _check(_shuffled_times(_field(5)), _grid(), 14)
    assert two[2] > 0


def test_repeated_detections():
    """Every detection three times (raw counts three times the distinct ones), and a cell that wraps an 8-bit counter."""
    cat = _field(6, noise=400)
    rep = lambda a: np.concatenate([a, a, a])  # noqa: E731
    _check(cases.catalog(rep(cat.x), rep(cat.y), rep(cat.epoch), cat.t, cat.ticks_per_hour), _grid(), 14)
    x = np.concatenate([cat.x, np.full(400, 500_000, np.int32)])
    y = np.concatenate([cat.y, np.full(400, 500_000, np.int32)])
    e = np.concatenate([cat.epoch, np.zeros(400, np.uint16)])
    _check(cases.catalog(x, y, e, cat.t, cat.ticks_per_hour), _grid(), 14)


def test_top_k_and_device_arrays():
    cat, grid = _field(7), _grid()
    full = _check(cat, grid, 14)[0]
    assert full[2] > 50
    top = _both(cat, grid, 14, max_candidates=50)[0]
    assert top[0] == full[0][:50 * 32]
    dev = [torch.from_numpy(a).cuda() for a in (cat.x, cat.y, cat.epoch.view(np.int16))]
    s = torch.cuda.Stream()
    res = sas.sas_stack(sas.Grid(grid), *dev, cat.t, cat.ticks_per_hour, 14, on_device=True, stream=s)
    assert res.candidates()[0].tobytes() == full[0]


@pytest.mark.parametrize("kind", ["ones", "wide", "zeros", "host"])
def test_weights(kind):
    """Weighted stacking through the windows: weights all one, over the whole range with repeated epochs in a bin, mostly
    zero, and from host arrays."""
    cat, grid = _field(9, movers=60), _grid()
    rep = np.concatenate
    x, y, e = rep([cat.x, cat.x]), rep([cat.y, cat.y]), rep([cat.epoch, cat.epoch])
    rng = np.random.default_rng(3)
    w = {"ones": np.ones(len(x)), "wide": rng.integers(0, 256, len(x)), "zeros": 200 * (rng.random(len(x)) < 0.1),
         "host": 20 + rng.integers(0, 60, len(x))}[kind].astype(np.uint8)
    s_min = {"ones": 16, "wide": 2600, "zeros": 1000, "host": 900}[kind]
    got = []
    for tiles in (dict(), dict(tile_kx=8, tile_ky=4)):
        o = sas.make_opts(**tiles)
        if kind == "host":
            res = sas.sas_stack_weighted(sas.Grid(grid), x, y, e, w, cat.t, cat.ticks_per_hour, s_min, opts=o)
        else:
            d = [torch.from_numpy(a).cuda() for a in (x, y, e.view(np.int16), w)]
            res = sas.sas_stack_weighted(sas.Grid(grid), *d, cat.t, cat.ticks_per_hour, s_min, opts=o, on_device=True)
        c, ids = res.candidates()
        got.append((c.tobytes(), ids.tobytes(), res.info()["n_pairs"]))
    assert got[0] == got[1]
    assert len(got[0][0]) > 0


def test_oracle():
    cat, grid = _field(8, width=700, height=900, noise=300), _grid(width=700, height=900)
    res = sas.stack_catalog(sas.Grid(grid), cat, 13)
    ref = oracle.stack(cat, grid, 13, threads=0)
    assert len(ref.cands) > 0
    assert_same(res, ref)


def _spot(cat, count, epochs):
    """cat without detections near (400, 700) px and with `count` there: 3 x 3 positions (5 x 5 for more) 3.6 px apart, each
    in every epoch until `count` is reached.  Cells of at most 3.6 px see no more than one of them an epoch."""
    keep = (np.abs(cat.x - 400_000) > 60_000) | (np.abs(cat.y - 700_000) > 60_000)
    k = np.arange(count)
    p, e, side = k // epochs, (k % epochs).astype(np.uint16), 3 if count <= 9 * epochs else 5
    x, y = (400_000 + 3600 * (p % side)).astype(np.int32), (700_000 + 3600 * (p // side)).astype(np.int32)
    return cases.catalog(np.r_[cat.x[keep], x], np.r_[cat.y[keep], y], np.r_[cat.epoch[keep], e], cat.t, cat.ticks_per_hour)


@pytest.mark.parametrize("epochs,count,two_levels", [(130, 256, True), (130, 257, True), (130, 1170, True), (250, 2000, True),
                                                     (250, 6250, False)])
def test_detections_in_one_window(epochs, count, two_levels):
    """Up to 256 detections of a window are listed by the first pass, up to 2048 by the second, and more send the field to
    the one-level search."""
    cat = _spot(_field(11, epochs=epochs, noise=40_000 // epochs, movers=20), count, epochs)
    two, one = _check(cat, _grid(), epochs // 3)
    assert two[2] > 0
    assert (two[3]["n_emitted"] != one[3]["n_emitted"]) == two_levels


def test_long_windows_with_weights():
    cat, grid = _spot(_field(12, epochs=130, noise=300, movers=20), 1170, 130), _grid()
    w = (20 + np.random.default_rng(4).integers(0, 60, len(cat.x))).astype(np.uint8)
    got = []
    for tiles in (dict(), dict(tile_kx=8, tile_ky=4)):
        res = sas.sas_stack_weighted(sas.Grid(grid), cat.x, cat.y, cat.epoch, w, cat.t, cat.ticks_per_hour, 2000,
                                     opts=sas.make_opts(**tiles))
        c, ids = res.candidates()
        got.append((c.tobytes(), ids.tobytes(), res.info()["n_pairs"], res.info()["n_emitted"]))
    assert got[0][:3] == got[1][:3] and len(got[0][0]) > 0
    assert got[0][3] != got[1][3]


def test_bright_movers_over_many_epochs():
    """Movers seen in nearly all of 255 epochs: with the noise around them their windows hold more than 256 detections."""
    r = W.FieldRecipe(1021, 1777, 255, 4.0, 500, 25, (0.5, 15.0), (1.0, 0.97))
    two, one = _check(W.make_catalog(r, 13), _grid(), 90)
    assert two[2] > 0 and two[3]["n_emitted"] != one[3]["n_emitted"]


def _pool(attribute):
    """An attribute of the device's stream-ordered pool."""
    import ctypes
    cu, pool, v = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    if attribute == "reset":
        assert cu.cuMemPoolSetAttribute(pool, 8, ctypes.byref(v)) == 0   # CU_MEMPOOL_ATTR_USED_MEM_HIGH
    else:
        assert cu.cuMemPoolGetAttribute(pool, {"used": 7, "high": 8}[attribute], ctypes.byref(v)) == 0
    return v.value


def test_a_low_threshold_search_does_not_size_the_window_list():
    """Super-bins emitted by a one-level search on a grid say nothing about the windows of the next search on it."""
    cat, grid = _field(10), sas.Grid(_grid())

    def peak():
        torch.cuda.synchronize()
        _pool("reset")
        before = _pool("used")
        sas.stack_catalog(grid, cat, 14).free()
        return _pool("high") - before
    alone = [peak(), peak()]
    low = sas.stack_catalog(grid, cat, 4, opts=sas.make_opts(superbin=3))  # one level
    assert low.info()["n_emitted"] > 1 << 20
    low.free()
    assert peak() <= max(alone) + (1 << 20)


def test_more_windows_and_candidates_than_their_lists_hold_at_first():
    """Many movers: more windows than noise would leave and more candidates than the key list's first 131072; both lists
    grow to what was counted."""
    cat = _field(14, movers=2500)
    two, one = _check(cat, _grid(), 14)
    assert two[2] > 1 << 17
    assert two[3]["n_emitted"] > (1 << 18) + cat.n and two[3]["n_emitted"] != one[3]["n_emitted"]


@pytest.mark.parametrize("used,per_epoch,two_levels", [(130, 1, True), (130, 4, True), (1, 70_000, False)])
def test_counters_that_wrap(used, per_epoch, two_levels):
    """Detections of one position in the first `used` epochs: within and above what a cell's 8-bit counter holds, and above
    what 16 bits and a window's list hold."""
    cat = _field(15, epochs=130, noise=300, movers=20)
    x, y = np.full(per_epoch * used, 400_100, np.int32), np.full(per_epoch * used, 700_100, np.int32)
    e = np.tile(np.arange(used, dtype=np.uint16), per_epoch)
    cat = cases.catalog(np.r_[cat.x, x], np.r_[cat.y, y], np.r_[cat.epoch, e], cat.t, cat.ticks_per_hour)
    two, one = _check(cat, _grid(), 40)
    assert two[2] > 0
    assert (two[3]["n_emitted"] != one[3]["n_emitted"]) == two_levels


def test_autotune_returns_the_two_level_search_where_it_is_faster():
    """sas_autotune's own combinations set tiles, which keep a search to one level."""
    cat, grid = _field(16, noise=2000), sas.Grid(_grid())
    d = [torch.from_numpy(a).cuda() for a in (cat.x, cat.y, cat.epoch.view(np.int16))]
    best, ms = sas.sas_autotune(grid, *d, cat.t, cat.ticks_per_hour, 22, reps=2)
    n = [sas.sas_stack(grid, *d, cat.t, cat.ticks_per_hour, 22, on_device=True, opts=o).info()["n_emitted"]
         for o in (best, sas.make_opts(), sas.make_opts(tile_kx=8, tile_ky=8))]
    assert n[0] == n[1] != n[2] and ms > 0
    one, _ = sas.sas_autotune(grid, *d, cat.t, cat.ticks_per_hour, 22, base=sas.make_opts(counter_bits=8), reps=1)
    assert one.superbin in (1, 2, 3, 4)


def test_tuning_cache_keeps_tiles_for_batches():
    """The cache's choices go to batches, which search in one level: they name tiles."""
    from paper_2509_26279_gb300 import tuning

    class F:
        pass

    f = F()
    f.cat, spec = _field(16, noise=2000), _grid()
    f.grid, f.E = sas.Grid(spec), f.cat.n_epochs
    f.dx, f.dy, f.de = (torch.from_numpy(a).cuda() for a in (f.cat.x, f.cat.y, f.cat.epoch.view(np.int16)))
    f.w = F()
    f.w.grid, f.w.n_min = spec, 22
    e = tuning.TuneCache().tune(f, reps=1)
    assert e["superbin"] in (1, 2, 3, 4) and e["tile_kx"] == 8


def test_the_info_names_the_counters_that_ran():
    """Weights are counted in 16 bits by a two-level search and, at this threshold, in 8 by the one-level plan."""
    cat, grid = _field(9, movers=60), sas.Grid(_grid())
    w = np.ones(len(cat.x), np.uint8)
    bits = [sas.sas_stack_weighted(grid, cat.x, cat.y, cat.epoch, w, cat.t, cat.ticks_per_hour, 16, opts=o).info()["counter_bits"]
            for o in (None, sas.make_opts(tile_kx=8, tile_ky=4))]
    assert bits == [16, 8]


@pytest.mark.parametrize("a,b", [(5, 3000), (333, 5999), (75 * 40 - 7, 75 * 40 + 1400), (2100, 75 * 83), (3, 1203)])
def test_lattice_ranges_of_a_denser_field(a, b):
    """Ranges that begin and end inside rows and inside groups, of a field dense enough that each is searched in two levels."""
    two, one = _check(_field(17, noise=2000), _grid(), 22, v_begin=a, v_end=b)
    assert two[2] > 0 and two[3]["n_emitted"] != one[3]["n_emitted"]


@pytest.mark.parametrize("epochs,n_min", [(11, 8), (128, 30), (150, 128), (255, 60)])
def test_epoch_counts_are_searched_in_two_levels(epochs, n_min):
    two, one = _check(_field(4, epochs=epochs, noise=60000 // epochs, movers=30), _grid(), n_min)
    assert two[3]["n_emitted"] != one[3]["n_emitted"]

"""The tiling of the step on moments (lbm_walk.cu: plan_walk), without a GPU: every CTA of a grid
writes one partial sum, so the grid has to fit the slots that the lattice's handle holds - as many as
the population step has CTAs - also for wide lattices of a few rows, and it has to cover the lattice."""
import ctypes
import os

import pytest

from paper_2301_12869_gb300 import _build, lbm

FP64, FP32 = 0, 1
NSM = 152


class WalkTiling(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("nx", "ny", "seg", "band_w", "nbands", "strip_h", "nstrips", "threads",
                                            "ctas", "zh")] + [("inv_n_total", ctypes.c_double)]


@pytest.fixture(scope="module")
def plan():
    if not os.path.exists(lbm.LIB_PATH):
        _build.build()
    lbm.load()
    fn = ctypes.CDLL(lbm.LIB_PATH)["_ZN3lbm9plan_walkEiiibiiPNS_10WalkTilingE"]
    fn.restype = ctypes.c_bool

    def call(precision, nx, ny, zh, slots):
        t = WalkTiling()
        ok = fn(precision, nx, ny, ctypes.c_bool(zh), NSM, slots, ctypes.byref(t))
        return ok, t

    return call


def slots_of(precision, nx, ny):
    """CTAs of the population step with its widest tile (the only one of Zou-He and thermal
    handles): 512 FP32 or 128 FP64 columns a band, one wave of at least one CTA an SM."""
    nbands = -(-nx // min(nx, 512 if precision == FP32 else 128))
    strips = max(1, min(ny, NSM // nbands))
    return nbands * -(-ny // -(-ny // strips))


@pytest.mark.parametrize("precision", [FP32, FP64])
@pytest.mark.parametrize("ny", [1, 2, 3, 4, 5, 8, 16, 33, 100, 1000])
@pytest.mark.parametrize("nx", [4, 60, 64, 508, 512, 516, 1024, 1924, 2048, 4096, 8192, 65536, 1 << 20])
def test_a_slot_for_every_cta(plan, precision, nx, ny):
    slots = slots_of(precision, nx, ny)
    ok, t = plan(precision, nx, ny, ny >= 3, slots)
    assert ok and 1 <= t.ctas <= slots, (t.ctas, slots)
    assert t.threads % 32 == 0 and 32 <= t.threads <= (512 if precision == FP32 else 256)
    # every band and strip has a segment, and they cover the lattice
    assert t.ctas * t.threads >= t.nbands * t.nstrips * t.seg
    assert t.nbands * t.band_w >= nx and t.band_w <= 2 * (t.seg - 2)
    assert t.nstrips * t.strip_h >= ny


@pytest.mark.parametrize("slots", [0, 1, 2])
def test_too_few_slots_are_reported(plan, slots):
    ok, t = plan(FP32, 4096, 8, True, slots)  # 69 warps of at most 16 a CTA
    assert not ok and t.ctas > slots


@pytest.mark.parametrize("precision, nx, ny, slots", [(FP32, 1024, 30, 60), (FP32, 424, 38, 38), (FP32, 308, 7, 7),
                                                      (FP64, 1256, 13, 130)])
def test_few_slots_take_more_warps_a_cta_before_taller_strips(plan, precision, nx, ny, slots):
    """A step's time is its strip's rows (and six of halo and rounding); warps beside each other cost
    little, so a grid that the slots bound keeps the strips it would have without them."""
    ok, free = plan(precision, nx, ny, True, 1 << 20)
    assert ok
    ok, t = plan(precision, nx, ny, True, slots)
    assert ok and t.ctas <= slots and t.strip_h <= free.strip_h + 2

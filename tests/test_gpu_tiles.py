"""The default tile follows the grid (choose_tile): the tile taken on each side
of one tile per SM, the same results as on the largest shape (bitwise for float
intensities, whose arithmetic does not depend on the tile; to rounding, 1e-12,
for double), the allocation-free step on each of its shapes, and the coupled
step, whose slabs are cut in multiples of the tile."""
import numpy as np
import pytest
import torch

import oracle
from paper_1403_6126_gb300 import workloads as wlmod

from _helpers import gpu_context, initial_state, rel_err
from test_zz_no_alloc import test_noalloc_step_equals_rt_step as noalloc_equals_rt_step

noalloc_equals_rt_step.__test__ = False
pytestmark = pytest.mark.gpu
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152


def _context(name, kw, precision):
    wl = wlmod.by_name(name, **kw)
    if precision == "fp32":
        wl = wlmod.rounded_to_float32(wl)
    n, w = oracle.angles.by_name(wl["angles"])
    ctx = gpu_context(wl, n, w, precision)
    ctx.set_intensity(initial_state(wl, len(w), precision))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    return ctx, wl


@pytest.mark.parametrize("name,kw,precision,tile,first", [
    ("slab1d", dict(n=64 * SMS, steps=0), "fp32", (64, 1, 1), (512, 1, 1)),
    ("slab1d", dict(n=64 * SMS + 1, steps=0), "fp32", (128, 1, 1), (512, 1, 1)),
    ("slab1d", dict(n=33, steps=0), "fp64", (64, 1, 1), (256, 1, 1)),
    ("slab1d", dict(n=128 * SMS + 1, steps=0), "fp64", (256, 1, 1), (256, 1, 1)),
    ("shadow2d", dict(nx=16 * SMS, ny=8, angles="s4", steps=0), "fp32", (16, 8, 1), (32, 16, 1)),
    ("shadow2d", dict(nx=16 * SMS + 1, ny=16, angles="s4", steps=0), "fp32", (16, 16, 1), (32, 16, 1)),
    ("shadow2d", dict(nx=8 * SMS, ny=7, angles="s4", steps=0), "fp64", (8, 8, 1), (16, 16, 1)),
    ("shadow2d", dict(nx=16 * SMS - 5, ny=9, angles="s4", steps=0), "fp64", (16, 16, 1), (16, 16, 1)),
    ("box3d", dict(n=9, angles="s4", steps=0), "fp32", (8, 8, 4), (16, 8, 4)),
])
def test_default_tile_and_its_results(name, kw, precision, tile, first):
    out = []
    for shape in (None, first):
        ctx, wl = _context(name, kw, precision)
        if shape is None:
            assert ctx.tile() == tile
        else:
            ctx.set_tile(*shape)
        for _ in range(2):
            ctx.step(0.0)
        ctx.sync()
        out.append((ctx.intensity(), ctx.moments()[0]))
        ctx.set_tile(0, 0, 0)
        assert ctx.tile() == tile
        ctx.close()
    for a, b in zip(*out):
        if precision == "fp32":
            np.testing.assert_array_equal(a, b)
        else:
            assert rel_err(a, b) <= 1e-12


@pytest.mark.parametrize("name,kw", [
    ("slab1d", dict(n=64 * SMS, steps=0)),
    ("slab1d", dict(n=64 * SMS + 1, steps=0)),
    ("slab1d", dict(n=128 * SMS + 1, steps=0)),
    ("slab1d", dict(n=256 * SMS + 1, steps=0)),
    ("shadow2d", dict(nx=16 * SMS, ny=8, angles="s4", steps=0)),
    ("shadow2d", dict(nx=16 * SMS + 1, ny=15, angles="s4", steps=0)),
])
def test_allocation_free_step_on_each_tile(name, kw):
    noalloc_equals_rt_step(name, kw)


@pytest.mark.parametrize("name,kw,precision", [
    ("slab1d", dict(n=1100, steps=0), "fp64"),
    ("slab1d", dict(n=1100, steps=0), "fp32"),
    ("shadow2d", dict(nx=40, ny=51, angles="s4", steps=0), "fp64"),
    ("shadow2d", dict(nx=40, ny=51, angles="s4", steps=0), "fp32"),
])
def test_coupled_step_cut_in_small_tiles(name, kw, precision):
    a, wl = _context(name, kw, precision)
    b, _ = _context(name, kw, precision)
    fields = wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"]
    dE, dM, T = a.step_coupled(0.0, *fields)
    b.set_material(*fields)
    b.step(0.0)
    dE2, dM2, T2 = b.sources()
    for x, y in ((dE, dE2), (dM, dM2), (T, T2), (a.intensity(), b.intensity())):
        np.testing.assert_array_equal(np.asarray(x).reshape(-1), np.asarray(y).reshape(-1))
    a.close()
    b.close()

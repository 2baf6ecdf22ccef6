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
    ("slab1d", dict(n=33, steps=0), "fp64", (32, 1, 1), (256, 1, 1)),
    ("slab1d", dict(n=32 * SMS, M=48, steps=0), "fp64", (32, 1, 1), (256, 1, 1)),
    ("slab1d", dict(n=32 * SMS + 1, steps=0), "fp64", (64, 1, 1), (256, 1, 1)),
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


@pytest.mark.parametrize("n,M", [(1, 1), (31, 2), (33, 7), (64, 8), (65, 9), (100, 48)])
@pytest.mark.parametrize("moving", [False, True])
def test_grouped_double_tile_matches_plain_tile(n, M, moving):
    # the 32-cell tile shares its angles out among four groups of threads
    wl = dict(wlmod.slab1d(n=n, steps=0))
    wl.update(hold_T=False, estimate_v=moving)
    rng = np.random.default_rng(n + M)
    v = np.zeros((3, n))
    if moving:
        v[:, n // 3:] = 0.1 * wl["C"] * (rng.random((3, n - n // 3)) - 0.5)
    nn = rng.normal(size=(M, 3))
    nn = np.ascontiguousarray(nn / np.sqrt((nn * nn).sum(1, keepdims=True)))
    w = rng.random(M) + 0.5
    w = w / w.sum()
    I = rng.random((M, n))
    out = []
    for tile in ((32, 1, 1), (64, 1, 1)):
        ctx = gpu_context(wl, nn, w, "fp64")
        ctx.set_tile(*tile)
        ctx.set_intensity(I)
        ctx.set_material(wl["rho"], wl["T"], v, wl["sa"], wl["ss"])
        for _ in range(3):
            ctx.step(0.0)
        ctx.sync()
        out.append([ctx.intensity(), *ctx.moments(), *ctx.sources()])
        ctx.close()
    scale = np.abs(out[1][1]).max()     # E: momentum and energy sources are differences of terms of P E / C, P E
    for k, (a, b) in enumerate(zip(*out)):
        tol = 1e-11 * max(np.abs(b).max(), scale)
        assert np.abs(a - b).max() <= tol, k

"""Accepted inputs near the ends of the number range, where a reciprocal or a
fast quotient is not defined although the division it stands for is."""
import numpy as np
import pytest

import oracle

from _helpers import gpu_context, rel_err, run_both

pytestmark = pytest.mark.gpu

P = 0


def _uniform(shape, rho, prat, sigma, T):
    N = int(np.prod(shape))
    dim = 3 if shape[0] > 1 else 2 if shape[1] > 1 else 1
    return dict(name="uniform", shape=shape, dim=dim, lo=(0.0, 0.0, 0.0), hi=(1.0, 1.0, 1.0), bc=((P, P),) * 3, C=10.0, P=prat,
                gamma=5.0 / 3.0, R=1.0, cfl=0.4, hold_T=False, estimate_v=False, steps=0, precision="fp32",
                rho=np.full(N, rho), T=np.full(N, T), v=np.zeros((3, N)), sa=np.full(N, sigma), ss=np.zeros(N),
                I0="isotropic_quarter_pi", inflow={}, angles="s4")


@pytest.mark.parametrize("shape", [(1, 1, 40), (1, 9, 12), (5, 4, 9)])
def test_float_temperature_solve_at_a_large_heat_capacity(shape):
    # rho R / (gamma - 1) = 1.5e38, above 2^126: the gas cools by a part in a
    # thousand or more, as in the oracle
    wl = _uniform(shape, 1e38, 1e35, 1.0, 3.2)
    n, w = oracle.angles.by_name("s4")
    g, o = run_both(wl, 3, "fp32", n=np.ascontiguousarray(n), w=np.ascontiguousarray(w))
    assert o["T"].max() < 3.2 - 1e-3
    assert rel_err(g["T"], o["T"]) <= 1e-5


@pytest.mark.parametrize("shape", [(1, 1, 40), (1, 9, 12), (5, 4, 9)])
def test_float_temperature_solve_at_a_subnormal_heat_capacity(shape):
    # without opacity nothing heats the gas: T stays as it is, and no cell fails
    wl = _uniform(shape, 1e-39, 1.0, 0.0, 1.0)
    n, w = oracle.angles.by_name("s4")
    ctx = gpu_context(wl, np.ascontiguousarray(n), np.ascontiguousarray(w), "fp32")
    ctx.set_intensity(np.full((len(w), wl["rho"].size), 1.0 / (4 * np.pi)))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    for _ in range(3):
        ctx.step(0.0)
    ctx.sync()
    np.testing.assert_array_equal(ctx.sources()[2].reshape(-1), wl["T"])
    ctx.close()


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 40), (1, 1, 20000), (1, 9, 12), (5, 4, 9)])
def test_double_step_at_a_subnormal_density(shape, moving):
    # without opacity nothing acts on the gas: T stays, the sources are zero
    wl = _uniform(shape, 1e-310, 1.0, 0.0, 1.0)
    wl.update(estimate_v=moving, v=np.full_like(wl["v"], 0.5 * moving))
    n, w = oracle.angles.by_name("s4")
    n, w = np.ascontiguousarray(n), np.ascontiguousarray(w)
    ctx = gpu_context(wl, n, w, "fp64")
    ctx.set_intensity(np.random.default_rng(4).random((len(w), wl["rho"].size)))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    for _ in range(3):
        ctx.step(0.0)
    ctx.sync()
    dE, dM, T = ctx.sources()
    np.testing.assert_array_equal(T.reshape(-1), wl["T"])
    assert not np.asarray(dE).any() and not np.asarray(dM).any()
    assert np.isfinite(ctx.intensity()).all()
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 1, 40), (1, 9, 12), (5, 4, 9)])
def test_double_slopes_of_tiny_intensities(shape):
    # products of differences near 1e-316, subnormal, are still positive: transport
    # as at the usual scale, but for the rounding of a product to 2^-1074, which
    # changes a slope s by at most 2^-28 / s or s / 4, so 2^-15 at most of the
    # intensity (a Courant number of 0.4 lets a fifth of that through); a slope
    # taken for zero shows in the second digit
    wl = _uniform(shape, 1.0, 1.0, 0.0, 1.0)
    wl["hold_T"] = True
    n, w = oracle.angles.by_name("s4")
    n, w = np.ascontiguousarray(n), np.ascontiguousarray(w)
    I = 1.0 + np.random.default_rng(8).random((len(w), wl["rho"].size))
    out = []
    for scale in (1.0, 2.0 ** -524):
        ctx = gpu_context(wl, n, w, "fp64")
        ctx.set_intensity(I * scale)
        ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
        ctx.step(0.0)
        ctx.sync()
        out.append(ctx.intensity() / scale)
        ctx.close()
    assert rel_err(out[1], out[0]) <= 1e-5

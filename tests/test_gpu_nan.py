"""A NaN in a saved state stays where the method puts it: the slopes beside it are
zero (no product of differences is positive), so one step spreads it to the
cells next to it and no further, as in the oracle."""
import numpy as np
import pytest

import oracle
from paper_1403_6126_gb300 import workloads as wlmod

from _helpers import gpu_context, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", [(1, 1, 45), (1, 11, 20), (9, 10, 11)])
def test_one_step_spreads_nan_to_the_next_cells(shape, precision, sign):
    rho, v, sa, ss = wlmod._gas_fields(shape, 100.0, 11, 2.0)
    dim = 3 if shape[0] > 1 else 2 if shape[1] > 1 else 1
    N = rho.size
    wl = dict(name="nan", shape=shape, dim=dim, lo=(0.0, 0.0, 0.0), hi=(1.0, 1.0, 1.0), bc=((0, 0),) * 3, C=100.0, P=100.0,
              gamma=5.0 / 3.0, R=1.0, cfl=0.4, hold_T=True, estimate_v=False, steps=0, precision=precision,
              rho=rho, T=np.ones(N), v=np.zeros((3, N)), sa=sa, ss=ss, I0="equilibrium", inflow={})
    if precision == "fp32":
        wl = wlmod.rounded_to_float32(wl)
    n, w = oracle.angles.by_name("s4")
    n, w = np.ascontiguousarray(n), np.ascontiguousarray(w)
    M = len(w)
    I = np.random.default_rng(6).random((M, N)).astype(np.float32).astype(np.float64)
    ctx = gpu_context(wl, n, w, precision)
    ctx.set_intensity(I)
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    buf = np.array(ctx.save_state())
    m, cell = 5, N // 2
    head = 64 + 8 * 6 * M     # the intensity as [M][N] doubles, or quads of floats per cell
    if precision == "fp64":
        buf[head:].view(np.uint8)[: 8 * M * N].view(np.float64).reshape(M, N)[m, cell] = sign * np.nan
    else:
        buf[head:][: 4 * M * N].view(np.float32).reshape(M // 4, N, 4)[m // 4, cell, m % 4] = sign * np.nan
    ctx.load_state(buf)
    I[m, cell] = sign * np.nan
    ctx.step(0.0)
    got = np.isnan(ctx.intensity())
    p = oracle_problem(wl, n, w)
    want = np.isnan(oracle.run(p, oracle.cfl_dt(p, wl["cfl"]), 1, I, wl["T"], wl["rho"], wl["v"], wl["sa"], wl["ss"])["I"])
    want = want.reshape(M, N)
    assert want.any(axis=0).sum() == 1 + 2 * dim
    np.testing.assert_array_equal(got.reshape(M, N), want)
    ctx.close()

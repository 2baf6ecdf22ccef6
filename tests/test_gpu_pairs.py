"""The float step on opposite pairs of angles (rt_step_sym.cuh): against the
FP64 oracle where it can go wrong (ragged tiles, unequal cell sides, open
faces, faces of exactly zero velocity, the smallest sets, the caller's own
order of the angles), with the bounds of the other float parity tests; a set
without opposite angles, which takes the quad kernel, beside it; and the saved
state, whose intensities stay in the caller's order."""
import numpy as np
import pytest

import oracle
from paper_1403_6126_gb300 import workloads as wlmod

from _helpers import field_err, flux_magnitude, gpu_context, initial_state, rel_err, run_both

pytestmark = pytest.mark.gpu

P, V, C, I = 0, 1, 2, 3


def _set(name, seed=0):
    if name == "two pairs":
        n = np.array([[0.6, 0.64, 0.48], [0.28, -0.96, 0.0]])
        return np.concatenate([n, -n]), np.array([0.2, 0.3, 0.2, 0.3])
    if name == "no pairs":
        n, w = oracle.angles.by_name("s4")
        w = w.copy()
        w[0] *= 1.5           # the opposite of angle 0 has another weight
        return n, w / w.sum()
    n, w = oracle.angles.by_name(name.split()[0])
    if name.endswith("shuffled"):
        p = np.random.default_rng(seed).permutation(len(w))
        n, w = n[p], w[p]
    return n, w


def _problem(shape, hi, bc, still):
    rho, v, sa, ss = wlmod._gas_fields(shape, 100.0, 11, 2.0)
    if still == "half":       # faces of exactly zero velocity beside moving ones
        v = v.reshape(3, *shape)
        v[..., : shape[2] // 2] = 0.0
        v = v.reshape(3, -1)
    if still == "all":
        v = np.zeros_like(v)
    N = rho.size
    T = 1.0 + 0.05 * np.random.default_rng(5).random(N)
    return dict(name="pairs", shape=shape, dim=3 if shape[0] > 1 else 2, lo=(0.0, 0.0, 0.0), hi=hi, bc=bc, C=100.0, P=100.0,
                gamma=5.0 / 3.0, R=1.0, cfl=0.4, hold_T=False, estimate_v=still != "all", steps=0, precision="fp32",
                rho=rho, T=T, v=v, sa=sa, ss=ss, I0="equilibrium",
                inflow={(0, 0): ("beam", 0.2, 0)} if bc[0][0] == I else {})


@pytest.mark.parametrize("angles,shape,hi,bc,still", [
    ("s2", (5, 9, 17), (1.0, 0.7, 0.4), ((P, P), (V, C), (C, V)), "no"),
    ("s4 shuffled", (4, 8, 8), (1.0, 1.0, 0.5), ((P, P),) * 3, "half"),
    ("s6", (1, 33, 20), (1.0, 1.2, 1.0), ((I, C), (V, V), (P, P)), "no"),
    ("s8 shuffled", (3, 5, 9), (0.9, 0.5, 0.3), ((I, V), (P, P), (C, C)), "half"),
    ("two pairs", (2, 3, 5), (1.0, 1.0, 1.0), ((V, C), (C, V), (P, P)), "no"),
    ("two pairs", (1, 1 + 16, 33), (1.0, 0.5, 1.0), ((P, P),) * 3, "half"),
    ("s4", (9, 8, 7), (1.0, 1.0, 1.0), ((I, C), (V, V), (P, P)), "all"),
    ("no pairs", (5, 9, 10), (1.0, 0.7, 0.4), ((P, P), (V, C), (C, V)), "no"),
])
def test_pair_step_matches_oracle(angles, shape, hi, bc, still):
    n, w = _set(angles)
    g, o = run_both(_problem(shape, hi, bc, still), 3, "fp32", n=np.ascontiguousarray(n), w=np.ascontiguousarray(w))
    wl = o["wl"]
    assert rel_err(g["E"], o["E"]) <= 1e-5
    assert field_err({"F": flux_magnitude(g["F"])}, {"F": flux_magnitude(o["F"]), "E": o["E"]}, "F", wl) <= 1e-5
    assert rel_err(g["T"], o["T"]) <= 1e-5
    for k in ("I", "P", "dMom", "dEgas"):
        assert field_err(g, o, k, wl) <= 1e-4, (k, field_err(g, o, k, wl))


@pytest.mark.parametrize("angles", ["s4", "s6 shuffled"])
def test_saved_state_is_in_the_callers_order(angles):
    n, w = _set(angles)
    n, w = np.ascontiguousarray(n), np.ascontiguousarray(w)
    wl = _problem((3, 5, 9), (1.0, 0.5, 0.3), ((I, C), (V, V), (P, P)), "no")
    M, N = len(w), 3 * 5 * 9
    ctx = gpu_context(wl, n, w, "fp32")
    ctx.set_intensity(np.random.default_rng(2).random((M, N)))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    buf = ctx.save_state()
    head = 64 + 8 * 6 * M      # header, inflow in double; then the intensity as quads of the caller's angles
    quads = np.frombuffer(buf, dtype=np.float32, offset=head, count=M * N).reshape(M // 4, N, 4).transpose(0, 2, 1)
    np.testing.assert_array_equal(quads.reshape(M, N), ctx.intensity().astype(np.float32))
    tail = np.frombuffer(buf[-4 * 6 * M:], dtype=np.float32).reshape(6, M)
    np.testing.assert_array_equal(tail[0], wlmod.inflow_values(wl["inflow"][(0, 0)], n).astype(np.float32))
    other = gpu_context(wl, n, w, "fp32", inflow=False)
    other.load_state(buf)
    for c in (ctx, other):
        c.step(0.0)
        c.sync()
    np.testing.assert_array_equal(other.intensity(), ctx.intensity())
    ctx.close()
    other.close()

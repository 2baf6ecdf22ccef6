"""The allocation-free step on opposite pairs against rt_step, for sets whose quads
lie on 8-byte words of the caller's layout (s6, s8, two pairs), for one with none
there (s4), and for one with both kinds in one launch.  Imported by
test_gpu_noalloc_pairs.py; run as a program it goes through the same cases with
the index-checking library (RT_BOUNDS_CHECK) and prints OK when no index was out
of range."""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

import torch  # noqa: E402

import oracle  # noqa: E402
import paper_1403_6126_gb300 as rt  # noqa: E402
from paper_1403_6126_gb300 import build as rtbuild  # noqa: E402
from paper_1403_6126_gb300 import workloads as wlmod  # noqa: E402
from _helpers import gpu_context  # noqa: E402
from test_gpu_pairs import C, I, P, V, _problem, _set  # noqa: E402
from test_zz_no_alloc import _structs, from_quads, to_quads  # noqa: E402

# which quads take 8-byte words
SETS = {"s6": "all", "s8": "all", "s4": "none", "two pairs": "all", "s6 mixed": "some"}
OPEN, PERIODIC = ((I, C), (V, C), (C, V)), ((P, P),) * 3
CASES = [
    ("s6", (1, 33, 45), OPEN, "half"),          # 16 x 8 tiles
    ("s8", (1, 99, 209), OPEN, "no"),           # 16 x 16
    ("s6 mixed", (1, 99, 209), PERIODIC, "no"),
    ("s6 mixed", (1, 20, 33), OPEN, "half"),
    ("two pairs", (1, 33, 45), OPEN, "no"),
    ("s6", (61, 45, 40), OPEN, "no"),           # 480 tiles: a CTA walks several
    ("s8", (5, 9, 17), OPEN, "half"),
    ("s6 mixed", (9, 10, 33), OPEN, "half"),
    ("s6 mixed", (61, 45, 40), PERIODIC, "no"),
    ("s4", (13, 9, 17), OPEN, "half"),
]


def angle_set(name):
    n, w = _set(name.split()[0] if name.endswith("mixed") else name)
    if name.endswith("mixed"):
        p = np.arange(len(w))
        p[:9] = np.random.default_rng(5).permutation(9)
        n, w = n[p], w[p]
    return np.ascontiguousarray(n), np.ascontiguousarray(w)


def words(n):
    """For each stored quad (n, n', -n, -n'), whether n, n' and -n, -n' are each
    one 8-byte word of the caller's layout."""
    left, pairs = list(range(len(n))), []
    while left:
        m = left.pop(0)
        at = next(l for l in left if np.array_equal(n[l].astype(np.float32), -n[m].astype(np.float32)))
        left.remove(at)
        pairs.append((m, at))
    quads = [(pairs[i][0], pairs[i + 1][0], pairs[i][1], pairs[i + 1][1]) for i in range(0, len(pairs), 2)]
    return [q[0] % 2 == 0 and q[1] == q[0] + 1 and q[2] % 2 == 0 and q[3] == q[2] + 1 for q in quads]


def check(name, shape, bc, still, steps=2):
    wl = wlmod.rounded_to_float32(_problem(shape, (1.0, 0.8, 0.6), bc, still))
    n, w = angle_set(name)
    N, M = int(np.prod(shape)), len(w)
    ctx = gpu_context(wl, n, w, "fp32")
    ctx.set_intensity(np.random.default_rng(M).random((M, N)).astype(np.float32).astype(np.float64))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    dt = ctx.cfl_dt()
    dev = torch.device("cuda", 0)
    f32 = lambda x: torch.tensor(np.asarray(x, dtype=np.float32).reshape(-1), device=dev)
    f64 = lambda x: torch.tensor(np.asarray(x, dtype=np.float64).reshape(-1), device=dev)
    Iq = [to_quads(ctx.intensity(), M, N, dev), torch.empty(M * N, dtype=torch.float32, device=dev)]
    E, F, Pr = ctx.moments()
    mom = [f64(np.concatenate([E.reshape(1, N), F.reshape(3, N), Pr.reshape(6, N)])), f64(np.zeros(10 * N))]
    rho, sa, ss, v, T = f32(wl["rho"]), f32(wl["sa"]), f32(wl["ss"]), f32(wl["v"]), f64(wl["T"])
    dE, dM = f64(np.zeros(N)), f64(np.zeros(3 * N))
    inflow = np.zeros((3, 2, M))
    for (axis, side), rule in wl["inflow"].items():
        inflow[axis, side] = wlmod.inflow_values(rule, n)
    g, a, o = _structs(wl, n, w)
    for k in range(steps):
        f = rt.rt_noalloc_fields()
        f.I_in, f.I_out = Iq[k % 2].data_ptr(), Iq[1 - k % 2].data_ptr()
        f.rho, f.sigma_a, f.sigma_s, f.v, f.T = (x.data_ptr() for x in (rho, sa, ss, v, T))
        f.mom_in, f.mom_out = mom[k % 2].data_ptr(), mom[1 - k % 2].data_ptr()
        f.dE_gas, f.dMom = dE.data_ptr(), dM.data_ptr()
        f.inflow = inflow.ctypes.data
        assert rt.rt_step_noalloc(g, a, wl["C"], wl["P"], o, dt, f) == 0
        ctx.step(dt)
        ctx.sync()
        out = mom[1 - k % 2].cpu().numpy().reshape(10, N)
        got = [from_quads(Iq[1 - k % 2], M, N), out[0], out[1:4], out[4:], dE.cpu().numpy(), dM.cpu().numpy(), T.cpu().numpy()]
        ref = [ctx.intensity(), *ctx.moments(), *ctx.sources()]
        for i, (x, y) in enumerate(zip(got, ref)):
            np.testing.assert_array_equal(np.asarray(x).reshape(-1), np.asarray(y).reshape(-1), err_msg="%d of step %d" % (i, k))
    ctx.close()


def main():
    rt.LIB_PATH = rtbuild.build(check=True)
    for case in CASES:
        check(*case)
        print("checked", *case, flush=True)
    print("OK", flush=True)


if __name__ == "__main__":
    main()

"""Child process of test_gpu_short_arrays.py: device arrays whose allocation ends
before the call's last element are refused (RT_E_CUDA) by every call that reads
or writes device arrays in place, as by the copies it replaces; allocations of
the exact length are taken.  One call per invocation, as an RT_E_CUDA may leave
the context unusable.  Every array here ends inside the 2 MiB page that holds
its start."""
import ctypes
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

import torch  # noqa: E402

import oracle  # noqa: E402
import paper_1403_6126_gb300 as rt  # noqa: E402
from paper_1403_6126_gb300 import workloads as wlmod  # noqa: E402
from _helpers import gpu_context  # noqa: E402

MIB = 1 << 20


def allocate(nbytes):
    assert MIB <= nbytes <= 2 * MIB      # pages of its own
    p = ctypes.c_uint64(0)
    assert ctypes.CDLL("libcuda.so.1").cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
    return p.value


def main(call, short):
    torch.zeros(1, device="cuda")
    n_grid = 51 if call != "intensity" else 26       # need: 1.01 MiB, or 8 angles of 0.13 MiB
    wl = wlmod.box3d(n=n_grid, angles="s2", steps=0)
    n, w = oracle.angles.by_name("s2")
    ctx = gpu_context(wl, np.ascontiguousarray(n), np.ascontiguousarray(w), "fp32", device_ptrs=True)
    N, M = n_grid ** 3, len(w)
    need = 8 * N * (M if call == "intensity" else 1)
    p = allocate(MIB if short else need)
    assert MIB < need < 2 * MIB
    dev = [torch.tensor(np.ascontiguousarray(wl[k]).reshape(-1), dtype=torch.float64, device="cuda")
           for k in ("rho", "T", "v", "sa", "ss")]
    ptr = [d.data_ptr() for d in dev]
    torch.cuda.synchronize()
    lib = rt.lib()
    if call == "material":
        assert ctypes.CDLL("libcuda.so.1").cuMemcpyDtoD_v2(ctypes.c_uint64(p), ctypes.c_uint64(ptr[1]),
                                                           ctypes.c_size_t(MIB if short else need)) == 0
        ptr[1] = p
    status = lib.rt_set_material(ctx.ctx, *ptr)
    if call != "material":
        assert status == rt.RT_OK
        if call == "intensity":
            status = lib.rt_get_intensity(ctx.ctx, p)
        else:
            out = [torch.empty(k * N, dtype=torch.float64, device="cuda").data_ptr() for k in (1, 3, 6)]
            if call == "moments":
                status = lib.rt_moments(ctx.ctx, p, out[1], out[2])
            else:
                status = lib.rt_sources(ctx.ctx, out[0], out[1], p)
    assert status == (rt.RT_E_CUDA if short else rt.RT_OK), (status, rt.rt_last_error())
    torch.cuda.synchronize()
    print("OK", flush=True)


if __name__ == "__main__":
    main(sys.argv[1], sys.argv[2] == "short")

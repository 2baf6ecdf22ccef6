"""Device arrays read and written in place (device_ptrs): the intensity comes out
bitwise as through the host path, for sets in every stored order, ragged angle
counts, zero and subnormal values, and an array off the 8-byte boundary; the
gas fields go in bitwise as from the host, a bad value is refused and leaves
the material as it was."""
import numpy as np
import pytest
import torch

import oracle
import paper_1403_6126_gb300 as rt
from paper_1403_6126_gb300 import workloads as wlmod

from _helpers import gpu_context

pytestmark = pytest.mark.gpu


def _angles(name):
    if name.startswith("random"):
        m = int(name.split()[1])
        n = np.random.default_rng(m).normal(size=(m, 3))
        return n / np.sqrt((n * n).sum(1, keepdims=True)), np.full(m, 1.0 / m)
    n, w = oracle.angles.by_name(name.split()[0])
    if name.endswith("shuffled"):
        p = np.random.default_rng(3).permutation(len(w))
        n, w = n[p], w[p]
    return np.ascontiguousarray(n), np.ascontiguousarray(w)


def _values(M, N):
    r = np.random.default_rng(M * N).random((M, N)).astype(np.float32).astype(np.float64)
    r.reshape(-1)[:: 7] = 0.0
    r.reshape(-1)[3:: 11] = float(np.float32(1e-40))
    r.reshape(-1)[5:: 13] *= float(np.float32(2.0 ** 60))
    return r


def _pair(name, n, w, precision, kw):
    wl = wlmod.by_name(name, **kw)
    dev = gpu_context(wl, n, w, precision, device_ptrs=True)
    return wl, dev, gpu_context(wl, n, w, precision)


@pytest.mark.parametrize("name,kw,angles,precision", [
    ("box3d", dict(n=9, angles="s4", steps=0), "s4 shuffled", "fp32"),
    ("box3d", dict(n=5, angles="s4", steps=0), "random 7", "fp32"),
    ("shadow2d", dict(nx=33, ny=21, angles="s4", steps=0), "s8", "fp32"),
    ("slab1d", dict(n=1, steps=0), "random 1", "fp32"),
    ("slab1d", dict(n=1021, steps=0), "random 9", "fp32"),
    ("shadow2d", dict(nx=33, ny=21, angles="s4", steps=0), "s4 shuffled", "fp64"),
])
@pytest.mark.parametrize("off", [0, 4])
def test_intensity_to_device_arrays(name, kw, angles, precision, off):
    n, w = _angles(angles)
    wl, dev, host = _pair(name, n, w, precision, kw)
    M, N = len(w), int(np.prod(wl["shape"]))
    I = _values(M, N)
    d = torch.tensor(I, device="cuda")
    dev.set_intensity(d)
    host.set_intensity(I)
    raw = torch.zeros(8 * M * N + 8, dtype=torch.uint8, device="cuda")
    assert rt.lib().rt_get_intensity(dev.ctx, raw.data_ptr() + off) == rt.RT_OK
    torch.cuda.synchronize()
    got = raw.cpu().numpy()[off:off + 8 * M * N].copy().view(np.float64).reshape(M, N)
    np.testing.assert_array_equal(got, host.intensity())
    np.testing.assert_array_equal(got, I)
    dev.close()
    host.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", ["cube", "flat"])
def test_fields_from_device_arrays(precision, shape):
    # "flat": cells of three different sides, and fewer cells than angles
    n, w = _angles("s8" if shape == "flat" else "s4")
    wl = dict(wlmod.by_name("box3d", n=9, angles="s4", steps=0))
    if shape == "flat":
        rho, v, sa, ss = wlmod._gas_fields((2, 3, 4), 100.0, 11, 2.0)
        wl.update(shape=(2, 3, 4), rho=rho, v=v, sa=sa, ss=ss, T=np.ones(24))
    dev = gpu_context(wl, n, w, precision, device_ptrs=True)
    host = gpu_context(wl, n, w, precision)
    f = [np.ascontiguousarray(wl[k]).reshape(-1) for k in ("rho", "T", "v", "sa", "ss")]
    d = [torch.tensor(x, dtype=torch.float64, device="cuda") for x in f]
    dev.set_material(*d)
    host.set_material(*f)
    for bad in range(5):
        b = [x.clone() for x in d]
        b[bad][-1] = float("nan")
        with pytest.raises(rt.RTError) as err:
            dev.set_material(*b)
        assert err.value.status == rt.RT_E_NONFINITE
    for x in d:
        x.zero_()           # the caller's arrays are free once the call has returned
    for c in (dev, host):
        for _ in range(2):
            c.step(0.0)
        c.sync()
    other = gpu_context(wl, n, w, precision)       # alpha comes back with a saved state
    other.load_state(host.save_state())
    for c in (dev, host, other):
        c.step(0.0)
        c.sync()
    M, N = len(w), len(f[0])
    I = torch.empty(M * N, dtype=torch.float64, device="cuda")
    rt.rt_get_intensity(dev.ctx, I)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(I.cpu().numpy().reshape(M, N), host.intensity())
    np.testing.assert_array_equal(other.intensity(), host.intensity())
    for c in (dev, host, other):
        c.close()


@pytest.mark.parametrize("want", [(1, 1, 1), (1, 0, 1), (0, 1, 0), (0, 0, 0)])
@pytest.mark.parametrize("off", [0, 4])
def test_moments_and_sources_to_device_arrays(want, off):
    n, w = _angles("s4")
    wl, dev, host = _pair("box3d", n, w, "fp32", dict(n=7, angles="s4", steps=0))
    N = int(np.prod(wl["shape"]))
    f = [np.ascontiguousarray(wl[k]).reshape(-1) for k in ("rho", "T", "v", "sa", "ss")]
    dev.set_material(*[torch.tensor(x, dtype=torch.float64, device="cuda") for x in f])
    host.set_material(*f)
    for c in (dev, host):
        c.step(0.0)
        c.sync()
    for call, sizes, ref in ((rt.lib().rt_moments, (1, 3, 6), host.moments()), (rt.lib().rt_sources, (1, 3, 1), host.sources())):
        raw = [torch.zeros(8 * k * N + 8, dtype=torch.uint8, device="cuda") for k in sizes]
        assert call(dev.ctx, *[r.data_ptr() + off if use else None for r, use in zip(raw, want)]) == rt.RT_OK
        torch.cuda.synchronize()
        for r, k, use, x in zip(raw, sizes, want, ref):
            got = r.cpu().numpy()
            if use:
                np.testing.assert_array_equal(got[off:off + 8 * k * N].copy().view(np.float64), np.asarray(x).reshape(-1))
            else:
                assert not got.any()
    dev.close()
    host.close()

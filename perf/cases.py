"""What the radiation-transfer library is measured on: calls that programs make through its public entry points.

A case is a dict of plain values.  `kind` says which program it stands for:
  run      a problem advanced on the device (rt_run), then its snapshot read: moments, temperature, intensity
  gas      a gas code on the device: every pass new fields (rt_set_material), one step, the sources back
  coupled  a gas code on the host: the same in one call with page-locked arrays (rt_step_coupled)
  batch    many small problems of uneven size in one persistent launch per step (rt_batch_step)
  serve    requests submitted to the serving loop together and collected (rt_submit, rt_server_wait, rt_poll)
  noalloc  one step on the caller's own device buffers (rt_step_noalloc)
and `medium` which of the paper's problems the fields are shaped like: "slab" (sec. 5.3), "shadow" (sec. 5.8),
"box" (the radiation-dominated moving medium of the sec. 6 setup), "open" (a static 3-D cloud between open faces).

Single-precision contexts hold float intensities and give results of float accuracy in double arrays; the programs
here keep those as float32.  Fields are drawn so that float32 holds them exactly.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1403_6126_gb300 as rt

PERIODIC, VACUUM, COPY, INFLOW = 0, 1, 2, 3
FOURPI = 4.0 * math.pi


def listed():
    return [
        # sec. 5.3 scattering atmosphere, 512 cells and 8 Gauss-Legendre angles in double, gas temperature held
        dict(name="slab_fp64", kind="run", medium="slab", prec="fp64", nx=512, ny=1, nz=1, angles="gl8", steps=100, hold=True),
        # sec. 5.8 shadow problem at its own size, beam through the left face, in float and in double
        dict(name="shadow", kind="run", medium="shadow", prec="fp32", nx=256, ny=128, nz=1, angles="s8", steps=50, hold=True),
        dict(name="shadow_fp64", kind="run", medium="shadow", prec="fp64", nx=256, ny=128, nz=1, angles="s8", steps=6, hold=True),
        # the sec. 6 performance setup: 128^3 cells, 80 angles, moving medium, gas temperature live
        dict(name="box3d", kind="run", medium="box", prec="fp32", nx=128, ny=128, nz=128, angles="s8", steps=8, hold=False),
        # a plane problem of the serving stream's size with moving gas
        dict(name="box2d", kind="run", medium="box", prec="fp32", nx=256, ny=256, nz=1, angles="s8", steps=20, hold=False),
        # a static cloud lit through one face, open on all others, ragged sides
        dict(name="open3d", kind="run", medium="open", prec="fp32", nx=75, ny=50, nz=61, angles="s6", steps=10, hold=False),
        # a gas code on the device around the step, new fields every step
        dict(name="gas_loop", kind="gas", medium="box", prec="fp32", nx=96, ny=80, nz=72, angles="s4", steps=1, hold=False),
        # a double-precision gas code on the host
        dict(name="coupled_fp64", kind="coupled", medium="box", prec="fp64", nx=48, ny=40, nz=36, angles="s4", steps=1, hold=False),
        # 512 uneven slabs and squares, one launch per step
        dict(name="batch", kind="batch", medium="slab", prec="fp32", count=512, steps=24, hold=False),
        # a burst of requests to the serving loop, plane and 3-D alternating
        dict(name="serve", kind="serve", medium="box", prec="fp32", count=8, steps=20, hold=False),
        # one step on the caller's buffers: the smallest call, and a ragged 3-D one with open faces
        dict(name="noalloc_small", kind="noalloc", medium="box", prec="fp32", nx=64, ny=48, nz=1, angles="s4", steps=1, hold=False),
        dict(name="noalloc_3d", kind="noalloc", medium="box", prec="fp32", nx=70, ny=64, nz=45, angles="s6", steps=1, hold=False, lit=True),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def angles():
        return rng.choice(["s2", "s4", "s6", "s8"])

    kind = rng.choice(["slab", "shadow", "box3d", "box3d", "box2d", "open", "gas", "coupled", "batch", "serve", "noalloc"])
    if kind == "slab":
        c = dict(kind="run", medium="slab", prec=rng.choice(["fp32", "fp64"]), nx=size(64, 4096), ny=1, nz=1,
                 angles="gl%d" % rng.choice([8, 16, 24, 32, 40, 48]), steps=2 * size(10, 50), hold=rng.random() < 0.5)
    elif kind == "shadow":
        p = rng.choice(["fp32", "fp32", "fp64"])
        c = dict(kind="run", medium="shadow", prec=p, nx=size(64, 320), ny=size(48, 200), nz=1, angles=angles(),
                 steps=2 * size(5, 25) if p == "fp32" else 2, hold=True)
    elif kind == "box3d":
        p = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        hi = 128 if p == "fp32" else 48
        c = dict(kind="run", medium="box", prec=p, nx=size(24, hi), ny=size(24, hi), nz=size(24, hi), angles=angles(),
                 steps=2 * rng.randint(1, 4), hold=False)
    elif kind == "box2d":
        c = dict(kind="run", medium="box", prec="fp32", nx=size(64, 512), ny=size(64, 512), nz=1, angles=angles(),
                 steps=2 * rng.randint(2, 10), hold=False)
    elif kind == "open":
        c = dict(kind="run", medium="open", prec="fp32", nx=size(24, 110), ny=size(24, 110), nz=size(24, 110),
                 angles=angles(), steps=2 * rng.randint(1, 5), hold=rng.random() < 0.3)
    elif kind == "gas":
        c = dict(kind="gas", medium="box", prec="fp32", nx=size(32, 128), ny=size(32, 128), nz=size(32, 128),
                 angles=angles(), steps=1, hold=False)
    elif kind == "coupled":
        c = dict(kind="coupled", medium="box", prec="fp64", nx=size(24, 64), ny=size(24, 64), nz=size(24, 48),
                 angles=rng.choice(["s2", "s4"]), steps=1, hold=False)
    elif kind == "batch":
        c = dict(kind="batch", medium="slab", prec="fp32", count=size(32, 512), steps=2 * rng.randint(2, 10), hold=False)
    elif kind == "serve":
        c = dict(kind="serve", medium="box", prec="fp32", count=rng.randint(3, 8), steps=rng.randint(8, 20), hold=False)
    else:
        three = rng.random() < 0.5
        c = dict(kind="noalloc", medium="box", prec="fp32", nx=size(24, 96 if three else 256), ny=size(24, 96 if three else 256),
                 nz=size(24, 64) if three else 1, angles=angles(), steps=1, hold=False, lit=rng.random() < 0.5)
    return c


# ---- inputs ------------------------------------------------------------------------------------------------------

_MU1 = {4: 0.3500212, 6: 0.2666355, 8: 0.2182179}     # level-symmetric first cosine (Carlson 1963)


def _angles(name):
    """Unit vectors [M, 3] and weights [M] (sum 1): level-symmetric "sN" or Gauss-Legendre "glM"."""
    if name.startswith("gl"):
        mu, w = np.polynomial.legendre.leggauss(int(name[2:]))
        return np.stack([mu, np.sqrt(1.0 - mu * mu), np.zeros_like(mu)], axis=1), w / w.sum()
    N = int(name[1:])
    L = N // 2
    if N == 2:
        lev = np.array([1.0 / math.sqrt(3.0)])
    else:
        m2 = _MU1[N] ** 2
        lev = np.sqrt(m2 + 2.0 * (1.0 - 3.0 * m2) / (N - 2) * np.arange(L))
    pts = [(i, j, L - 1 - i - j) for i in range(L) for j in range(L - i)]
    keys = [tuple(sorted(p)) for p in pts]
    kinds = list(dict.fromkeys(keys))
    # one weight per kind of point: the normalisation and the even moments <mu^2k> = 1/(2k+1), k = 2, 3, ...
    A = np.zeros((len(kinds), len(kinds)))
    for p, k in zip(pts, keys):
        for r in range(len(kinds)):
            A[r, kinds.index(k)] += 1.0 if r == 0 else lev[p[0]] ** (2 * (r + 1))
    b = np.array([0.125 if r == 0 else 0.125 / (2 * (r + 1) + 1) for r in range(len(kinds))])
    wk = np.linalg.solve(A, b)
    n, w = [], []
    for s in range(8):
        sg = [-1.0 if s & (4 >> d) else 1.0 for d in range(3)]
        for p, k in zip(pts, keys):
            v = np.array([sg[d] * lev[p[d]] for d in range(3)])
            n.append(v / np.linalg.norm(v))
            w.append(wk[kinds.index(k)])
    w = np.array(w)
    return np.array(n), w / w.sum()


def _smooth(gen, shape, kmax):
    """Unit-variance Gaussian random field, P(k) ~ k^-2 on 1 <= |k| <= kmax (box units), on the device of gen."""
    dev = gen.device
    k = [torch.fft.fftfreq(s, device=dev, dtype=torch.float64) * s for s in shape]
    K = torch.sqrt(k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2)
    amp = torch.where((K >= 1.0) & (K <= kmax), 1.0 / K.clamp(min=1.0), torch.zeros_like(K))
    noise = torch.randn(shape, generator=gen, device=dev, dtype=torch.float64)
    f = torch.fft.ifftn(torch.fft.fftn(noise) * amp).real
    f = f - f.mean()
    return f / f.std()


def _f32(x):
    return x.to(torch.float32).to(torch.float64)


def _problem(case, seed):
    """Grid, parameters and gas fields (float64 tensors of float32 values, [N] and [3, N]) of one problem."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dim = 3 if nz > 1 else 2 if ny > 1 else 1
    N = nx * ny * nz
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 13)
    shape = (nz, ny, nx)
    n, w = _angles(case["angles"])
    M = len(w)
    p = dict(dim=dim, shape=shape, N=N, M=M, n=n, w=w, hold=bool(case["hold"]), inflow={}, lo=(0.0, 0.0, 0.0),
             hi=(1.0, ny / nx if dim >= 2 else 1.0, nz / nx if dim >= 3 else 1.0), bc=((PERIODIC, PERIODIC),) * 3)
    one = torch.ones(N, device=dev, dtype=torch.float64)

    def rand(lo, hi):
        return _f32(10.0 ** (lo + (hi - lo) * torch.rand(N, generator=gen, device=dev, dtype=torch.float64)))

    nt = torch.tensor(n, device=dev)
    if case["medium"] == "box":
        kmax = max(1.0, min(16.0, min(s for s in shape if s > 1) / 4.0))
        C = 100.0
        v = torch.stack([_smooth(gen, shape, kmax).reshape(N) for _ in range(3)])
        speed = v.square().sum(0).sqrt()
        want = (0.05 * C * speed / speed.square().mean().sqrt()).clamp(0.01 * C, 0.1 * C)
        rho = torch.exp(0.5 * _smooth(gen, shape, kmax).reshape(N) - 0.125)
        T = 1.0 + 0.05 * torch.tanh(_smooth(gen, shape, kmax).reshape(N))
        p.update(C=C, P=100.0, cfl=0.4, est=True, rho=_f32(rho), T=_f32(T), v=_f32(v * (want / speed.clamp(min=1e-300))),
                 sa=rand(0.0, 3.0), ss=rand(0.0, 3.0))
        J = (1.0 + 0.1 * torch.tanh(_smooth(gen, shape, kmax).reshape(N))) / FOURPI
        if case.get("lit"):          # a piece of the medium between open faces, lit from the left
            p["bc"] = ((INFLOW, COPY), (VACUUM, COPY), (PERIODIC, PERIODIC))
            p["inflow"] = {(0, 0): np.where(n[:, 0] > 0, 1.2 / FOURPI, 0.0)}
    elif case["medium"] == "slab":
        p.update(C=10.0, P=1.0, cfl=0.5 if dim == 1 else 0.4, est=False, rho=one.clone(), T=one.clone(),
                 v=torch.zeros(3, N, device=dev, dtype=torch.float64), sa=_f32(0.01 * one), ss=rand(-1.0, 2.0),
                 bc=((COPY, VACUUM), (PERIODIC, PERIODIC), (PERIODIC, PERIODIC)))
        x = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) / nx
        J = (one.reshape(shape) * (1.0 - 0.8 * x)).reshape(N) / FOURPI
    else:  # a cloud in a thin medium at rest, a beam through the left face; "open": 3-D, all other faces open
        x = [(torch.arange(s, device=dev, dtype=torch.float64) + 0.5) / s - 0.5 for s in (nx, ny, nz)]
        r = x[0][None, None, :] ** 2 / 0.01 + x[1][None, :, None] ** 2 / 0.01
        if dim == 3:
            r = r + x[2][:, None, None] ** 2 / 0.01
        rho = (1.0 + 9.0 / (1.0 + torch.exp((10.0 * (r - 1.0)).clamp(max=200.0)))).expand(shape).reshape(N)
        rho = _f32(rho * torch.exp(0.05 * torch.randn(N, generator=gen, device=dev, dtype=torch.float64)))
        T = _f32(1.0 / rho)
        p.update(C=10.0, P=1.0, cfl=0.4, est=False, rho=rho, T=T, v=torch.zeros(3, N, device=dev, dtype=torch.float64),
                 sa=_f32(T ** -3.5 * rho ** 2),
                 ss=_f32(0.1 * rho) if case["medium"] == "open" else torch.zeros_like(rho),
                 bc=((INFLOW, COPY), (VACUUM, VACUUM), (VACUUM, COPY) if dim == 3 else (PERIODIC, PERIODIC)))
        beam = np.where(n[:, 0] > 0, 10.0, 0.0)
        p["inflow"] = {(0, 0): beam}
        J = T ** 4 / FOURPI
    # the intensity of a problem under way: a dipole around J, and behind an open face the beam on its first cells
    aniso = torch.stack([torch.tanh(_smooth(gen, shape, 4.0).reshape(N)) for _ in range(3)]) * 0.25
    if dim < 3:
        aniso[dim:] = 0.0
    Im = J * (1.0 + nt @ aniso)
    if case["medium"] in ("shadow", "open"):
        front = (torch.arange(nx, device=dev) < 0.2 * nx).expand(shape).reshape(N)
        Im = torch.where(front & (nt[:, 0:1] > 0), 10.0 * torch.exp(-0.1 * p["sa"] / nx) + 0.0 * Im, Im)
    p["I"] = _f32(Im)
    h = [(p["hi"][d] - p["lo"][d]) / s for d, s in enumerate((nx, ny, nz))]
    p["dx"] = [h[d] if d < dim else 1.0 for d in range(3)]
    p["dt"] = p["cfl"] * min(h[:dim]) / p["C"]
    return p


def _members(case, seed):
    """The problems of a batch (slabs and squares of the atmosphere, sec. 5.3) or of a burst of requests (boxes)."""
    rng = np.random.default_rng(1000 + int(case["count"]))      # sizes belong to the case, fields to the seed
    out = []
    for i in range(case["count"]):
        if case["kind"] == "batch":
            if i % 2 == 0:
                c = dict(nx=int(round(np.exp(rng.uniform(np.log(64), np.log(4096))))), ny=1, nz=1,
                         angles="gl%d" % rng.choice([8, 16, 24, 32, 40, 48]))
            else:
                c = dict(nx=int(round(np.exp(rng.uniform(np.log(32), np.log(256))))),
                         ny=int(round(np.exp(rng.uniform(np.log(32), np.log(256))))), nz=1, angles=str(rng.choice(["s2", "s4", "s6"])))
        else:
            side = int(rng.choice([64, 96, 128, 192])) if i % 2 == 0 else int(rng.choice([32, 48, 64]))
            c = dict(nx=side, ny=side, nz=1 if i % 2 == 0 else side, angles=str(rng.choice(["s4", "s8"])))
        out.append((dict(c, kind=case["kind"], medium=case["medium"], hold=case["hold"], prec="fp32"), int(seed) * 1009 + i))
    return out


# ---- programs ----------------------------------------------------------------------------------------------------

def _context(p, prec, **kw):
    ctx = rt.Context(p["shape"], p["n"], p["w"], p["C"], p["P"], dim=p["dim"], lo=p["lo"], hi=p["hi"], bc=p["bc"],
                     precision=rt.RT_FP64 if prec == "fp64" else rt.RT_FP32, cfl=p["cfl"], hold_T=p["hold"],
                     estimate_v=p["est"], **kw)
    for (axis, side), val in p["inflow"].items():
        ctx.set_inflow(axis, side, val)
    return ctx


_stream = []


def _own_stream():
    """The one stream that a program of this process keeps its contexts on (a graph cannot be captured on the default one)."""
    if not _stream:
        _stream.append(torch.cuda.Stream())
    return _stream[0]


class _Program:
    """What a program keeps between calls; released when it is dropped."""

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if getattr(self, "server", None):
                rt.rt_server_destroy(self.server)
            if getattr(self, "batch", None):
                rt.rt_batch_destroy(self.batch)
            for c in getattr(self, "ctxs", []):
                c.close()
        except Exception:
            pass


def _structs(p, prec):
    g = rt.rt_grid()
    g.dim = p["dim"]
    for d in range(3):
        g.n[d], g.lo[d], g.hi[d] = p["shape"][2 - d], p["lo"][d], p["hi"][d]
        g.bc[d][0], g.bc[d][1] = p["bc"][d]
    a = rt.rt_angles()
    keep = (np.ascontiguousarray(p["n"]), np.ascontiguousarray(p["w"]))
    DP = ctypes.POINTER(ctypes.c_double)
    a.m, a.n, a.w = p["M"], keep[0].ctypes.data_as(DP), keep[1].ctypes.data_as(DP)
    o = rt.rt_options_default()
    o.precision = rt.RT_FP64 if prec == "fp64" else rt.RT_FP32
    o.cfl, o.hold_T, o.estimate_v = p["cfl"], int(p["hold"]), int(p["est"])
    return g, a, o, keep


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda")
    if kind == "batch":
        stream = _own_stream()
        stream.wait_stream(torch.cuda.current_stream())
        b = rt.rt_batch_create(stream.cuda_stream)
        ctxs, total = [], 0
        for c, s in _members(case, seed):
            p = _problem(c, s)
            torch.cuda.synchronize()
            ctx = _context(p, "fp32", device_ptrs=True, stream=stream.cuda_stream)
            ctx.set_intensity(p["I"])
            ctx.set_material(p["rho"], p["T"], p["v"], p["sa"], p["ss"])
            stream.synchronize()
            rt.rt_batch_add(b, ctx.ctx)
            ctxs.append(ctx)
            total += p["N"]
        out = torch.empty(10 * total, dtype=torch.float64, device=dev)
        views, o = [], 0
        for ctx in ctxs:
            n = ctx.N
            views.append((ctx.ctx, out[o:o + n], out[total + 3 * o:total + 3 * (o + n)], out[4 * total + 6 * o:4 * total + 6 * (o + n)]))
            o += n
        return _Program(kind=kind, steps=case["steps"], batch=b, ctxs=ctxs, stream=stream, out=out, views=views, total=total)
    if kind == "serve":
        reqs = []
        for c, s in _members(case, seed):
            p = _problem(c, s)
            f = {k: np.ascontiguousarray(p[k].cpu().numpy()) for k in ("rho", "T", "v", "sa", "ss")}
            reqs.append((p, f, _structs(p, "fp32"), np.empty(p["N"]), np.empty((3, p["N"])), np.empty((6, p["N"]))))
        opts = rt.rt_options_default()
        opts.hold_T, opts.estimate_v, opts.cfl = int(case["hold"]), 1, 0.4
        return _Program(kind=kind, steps=case["steps"], server=rt.rt_server_create(64 << 30, opts), reqs=reqs)
    p = _problem(case, seed)
    torch.cuda.synchronize()
    N, M = p["N"], p["M"]
    if kind == "noalloc":
        g, a, o, keep = _structs(p, "fp32")
        Q = (M + 3) // 4
        Iq = torch.zeros(4 * Q, N, dtype=torch.float32, device=dev)
        Iq[:M] = p["I"].float()
        I0 = Iq.reshape(Q, 4, N).permute(0, 2, 1).contiguous().reshape(-1)
        w, n = torch.tensor(p["w"], device=dev), torch.tensor(p["n"], device=dev)
        W = torch.stack([w, *(w * n[:, d] for d in range(3)), *(w * n[:, d] * n[:, d] for d in range(3)),
                         w * n[:, 0] * n[:, 1], w * n[:, 0] * n[:, 2], w * n[:, 1] * n[:, 2]])
        mom = (FOURPI * (W @ p["I"])).reshape(-1)
        # two buffer sets: moments (10 N), energy source (N), momentum source (3 N)
        res = [torch.cat([mom, torch.zeros(4 * N, dtype=torch.float64, device=dev)]) for _ in range(2)]
        inflow = np.zeros((3, 2, M))
        for (axis, side), val in p["inflow"].items():
            inflow[axis, side] = val
        f32 = {k: p[k].float().contiguous() for k in ("rho", "sa", "ss", "v")}
        return _Program(kind=kind, structs=(g, a, o, keep), p=p, I=[I0, torch.zeros_like(I0)], res=res, T=p["T"].clone(),
                        inflow=inflow, mat=f32, turn=0, N=N)
    if kind == "coupled":
        ctx = _context(p, case["prec"])
        ctx.set_intensity(p["I"].cpu().numpy())
        host = {}
        for k in ("rho", "T", "v", "sa", "ss"):
            host[k] = torch.empty(p[k].shape, dtype=torch.float64, pin_memory=True)
            host[k].copy_(p[k])
        out = [torch.empty(s, dtype=torch.float64, pin_memory=True) for s in ((N,), (3, N), (N,))]
        torch.cuda.synchronize()
        ctx.set_material(*(host[k].numpy() for k in ("rho", "T", "v", "sa", "ss")))
        return _Program(kind=kind, ctxs=[ctx], dt=p["dt"], host=host, out=out)
    stream = _own_stream()
    ctx = _context(p, case["prec"], device_ptrs=True, stream=stream.cuda_stream)
    ctx.set_intensity(p["I"])
    ctx.set_material(p["rho"], p["T"], p["v"], p["sa"], p["ss"])
    stream.synchronize()
    buf = torch.empty((5 if kind == "gas" else 11) * N, dtype=torch.float64, device=dev)
    if kind == "gas":
        other = dict(p, rho=_f32(p["rho"] * 1.03), T=_f32(p["T"] * 0.99), v=_f32(p["v"] * 0.98))
        p.pop("I"), other.pop("I")
        return _Program(kind=kind, ctxs=[ctx], stream=stream, dt=p["dt"], N=N, buf=buf, sets=[p, other], turn=0)
    p.pop("I")
    I = torch.empty(M, N, dtype=torch.float64, device=dev)
    return _Program(kind=kind, ctxs=[ctx], stream=stream, dt=p["dt"], N=N, buf=buf, I=I, steps=case["steps"], single=case["prec"] == "fp32")


def run(s):
    if s.kind == "run":
        c, N, b = s.ctxs[0], s.N, s.buf
        with torch.cuda.stream(s.stream):
            c.run(s.dt, s.steps)
            rt.rt_moments(c.ctx, b[:N], b[N:4 * N], b[4 * N:10 * N])
            rt.rt_sources(c.ctx, None, None, b[10 * N:])
            rt.rt_get_intensity(c.ctx, s.I)
            x, I = (b.float(), s.I.float()) if s.single else (b, s.I)
        return dict(E=x[:N], F=x[N:4 * N], P=x[4 * N:10 * N], T=x[10 * N:], I=I)
    if s.kind == "gas":
        c, N, b = s.ctxs[0], s.N, s.buf
        f = s.sets[s.turn % 2]
        s.turn += 1
        with torch.cuda.stream(s.stream):
            c.set_material(f["rho"], f["T"], f["v"], f["sa"], f["ss"])
            c.step(s.dt)
            rt.rt_sources(c.ctx, b[:N], b[N:4 * N], b[4 * N:])
            x = b.float()
        return dict(dE=x[:N], dM=x[N:4 * N], T=x[4 * N:])
    if s.kind == "coupled":
        h = s.host
        s.ctxs[0].step_coupled(s.dt, *(h[k].numpy() for k in ("rho", "T", "v", "sa", "ss")), *(o.numpy() for o in s.out))
        return dict(dE=s.out[0], dM=s.out[1], T=s.out[2])
    if s.kind == "batch":
        t = s.total
        with torch.cuda.stream(s.stream):
            rt.rt_batch_step(s.batch, s.steps)
            for c, E, F, P in s.views:
                rt.rt_moments(c, E, F, P)
            x = s.out.float()
        return dict(E=x[:t], F=x[t:4 * t], P=x[4 * t:])
    if s.kind == "serve":
        tickets = []
        for p, f, (g, a, _, _), *_ in s.reqs:
            tickets.append(rt.rt_submit(s.server, g, a, p["C"], p["P"], f["rho"], f["T"], f["v"], f["sa"], f["ss"], s.steps))
        out = []
        for ticket, (_, _, _, E, F, P) in zip(tickets, s.reqs):
            rt.rt_server_wait(s.server, ticket)
            rt.rt_poll(s.server, ticket, E, F, P)
            out.append([E.astype(np.float32), F.astype(np.float32), P.astype(np.float32)])
        return out
    # noalloc: the caller's buffers in turn
    g, a, o, _ = s.structs
    i, j, N = s.turn % 2, (s.turn + 1) % 2, s.N
    s.turn += 1
    f = rt.rt_noalloc_fields()
    f.I_in, f.I_out = s.I[i].data_ptr(), s.I[j].data_ptr()
    f.rho, f.sigma_a, f.sigma_s, f.v = (s.mat[k].data_ptr() for k in ("rho", "sa", "ss", "v"))
    f.T, f.mom_in, f.mom_out = s.T.data_ptr(), s.res[i].data_ptr(), s.res[j].data_ptr()
    f.dE_gas, f.dMom = s.res[j][10 * N:].data_ptr(), s.res[j][11 * N:].data_ptr()
    f.inflow = s.inflow.ctypes.data
    rt.rt_step_noalloc(g, a, s.p["C"], s.p["P"], o, s.p["dt"], f, want_failures=False)
    x = s.res[j].float()
    return dict(I=s.I[j], E=x[:N], F=x[N:4 * N], P=x[4 * N:10 * N], dE=x[10 * N:11 * N], dM=x[11 * N:], T=s.T.float())


# ---- what a pass cannot do without ---------------------------------------------------------------------------------

def _step_work(N, M, dim, prec, moving):
    """Bytes and operations of one step: the intensity read and written, rho, sigma_a, sigma_s, v, T in, E, F and P_dd in
    (velocity), the ten moments, T and four sources out; per cell and angle an axis costs about 16 operations of van
    Leer transport, and as many again for the velocity term, the implicit steps and the quadrature 40 to 75."""
    s = 8 if prec == "fp64" else 4
    return (N * (2 * M * s + 6 * s + 8 + (56 if moving else 0) + 15 * 8),
            N * M * (dim * (32 if moving else 16) + (75 if moving else 40)))


def work(case):
    cases = [c for c, _ in _members(case, 0)] if case["kind"] in ("batch", "serve") else [case]
    by = fl = 0
    for c in cases:
        N, M = c["nx"] * c["ny"] * c["nz"], len(_angles(c["angles"])[1])
        dim = 3 if c["nz"] > 1 else 2 if c["ny"] > 1 else 1
        b, f = _step_work(N, M, dim, c["prec"], c["medium"] == "box" or case["kind"] == "noalloc")
        by, fl = by + b * case["steps"], fl + f * case["steps"]
        if case["kind"] == "run":        # the snapshot's intensity as well
            by += N * M * (8 if c["prec"] == "fp64" else 4)
    return {"bytes": float(by), "flops": float(fl)}


# ---- the same in 64 bits, in plain torch -----------------------------------------------------------------------------

def _pad(x, axis, n, kinds, width):
    """x with `width` mapped cells beyond each end of an axis (periodic image, else the nearest cell)."""
    i = torch.arange(-width, n + width, device=x.device)
    i = i % n if kinds[0] == PERIODIC else i.clamp(0, n - 1)
    return x.index_select(axis, i)


def _vanleer(q, axis):
    """Harmonic-mean limited slope of every inner cell along an axis."""
    d = torch.diff(q, dim=axis)
    k = d.shape[axis]
    a, b = d.narrow(axis, 0, k - 1), d.narrow(axis, 1, k - 1)
    pr = a * b
    return torch.where(pr > 0, 2.0 * pr / torch.where(pr > 0, a + b, torch.ones_like(pr)), torch.zeros_like(pr))


def _transport(p, I, J, v, st, nt, lo, hi):
    """Delta F of angles lo..hi: I [m, nz, ny, nx], one unsplit step."""
    C, dt = p["C"], p["dt"]
    n = nt[lo:hi]
    m = hi - lo
    dF = torch.zeros_like(I)
    for d in range(p["dim"]):
        ax, N = 2 - d, p["shape"][2 - d]
        kinds, dx = p["bc"][d], p["dx"][d]
        mu = n[:, d].reshape(m, 1, 1, 1)
        Ip = _pad(I, ax + 1, N, kinds, 2).clone()
        for side in range(2):
            if kinds[side] in (VACUUM, INFLOW):
                coming = (n[:, d] > 0) if side == 0 else (n[:, d] < 0)
                val = torch.zeros(m, device=I.device, dtype=I.dtype)
                if kinds[side] == INFLOW and (d, side) in p["inflow"]:
                    val = torch.tensor(p["inflow"][(d, side)][lo:hi], device=I.device, dtype=I.dtype)
                g = Ip.narrow(ax + 1, 0 if side == 0 else N + 2, 2)
                g.copy_(torch.where(coming.reshape(m, 1, 1, 1), val.reshape(m, 1, 1, 1), g))
        w = 3.0 * _pad(J, ax, N, kinds, 2) * _pad(v, ax + 1, N, kinds, 2)
        IV = torch.einsum("md,dzyx->mzyx", n, w)
        It = Ip - IV / C
        al = _pad((torch.sqrt(-torch.expm1(-(10.0 * dx * st) ** 2) / ((10.0 * dx * st) ** 2).clamp(min=1e-300))), ax, N, kinds, 1)
        tau = _pad((10.0 * dx * st) ** 2, ax, N, kinds, 1)
        al = torch.where(tau < 1e-12, torch.ones_like(al), al)
        vd = _pad(v[d], ax, N, kinds, 1)
        af = 0.5 * (al.narrow(ax, 0, N + 1) + al.narrow(ax, 1, N + 1))
        vf = 0.5 * (vd.narrow(ax, 0, N + 1) + vd.narrow(ax, 1, N + 1))
        sI, sV = _vanleer(It, ax + 1), _vanleer(IV, ax + 1)
        left = lambda x, o: x.narrow(ax + 1, o, N + 1)  # noqa: E731
        nu = af * C * mu.abs() * dt / dx
        L = left(It, 1) + 0.5 * (1.0 - nu) * left(sI, 0)
        R = left(It, 2) - 0.5 * (1.0 - nu) * left(sI, 1)
        flux = 0.5 * C * mu * (L + R) + 0.5 * C * mu.abs() * af * (L - R)
        hv = 0.5 * (1.0 - vf.abs() * dt / dx)
        Lv = left(IV, 1) + hv * left(sV, 0)
        Rv = left(IV, 2) - hv * left(sV, 1)
        wl = torch.where(vf > 0, 1.0, torch.where(vf < 0, 0.0, 0.5))
        flux = flux + mu * (wl * Lv + (1.0 - wl) * Rv)
        dF -= dt / dx * torch.diff(flux, dim=ax + 1)
    return dF


def _step64(p, I, mom, T, f, nt, wt):
    """One step: I [M, N], mom [10, N], T [N], fields f; returns the new I, mom, T and the sources."""
    C, P, dt, M, N, shape = p["C"], p["P"], p["dt"], p["M"], p["N"], p["shape"]
    rho, v, sa, ss = f["rho"], f["v"], f["sa"], f["ss"]
    st = sa + ss
    grid = lambda x: x.reshape(x.shape[:-1] + shape)  # noqa: E731
    dF = torch.empty_like(I)
    chunk = max(1, min(M, (1 << 24) // N))
    for lo in range(0, M, chunk):
        hi = min(M, lo + chunk)
        dF[lo:hi] = _transport(p, grid(I[lo:hi]), grid(mom[0] / FOURPI), grid(v), grid(st), nt, lo, hi).reshape(hi - lo, N)
    vt = v
    if p["est"]:
        h = 0.5 * dt * st
        vt = torch.stack([(rho * v[d] + h * (C * rho * v[d] + P * mom[1 + d])) / (rho + h * (C * rho + P * (mom[0] + mom[4 + d]) / C))
                          for d in range(3)])
    v2 = vt.square().sum(0)
    W = wt.reshape(M, 1)
    vn = nt @ vt
    scat = (ss > sa).to(I.dtype)
    # absorption and the gas energy (sec. 4.3)
    A1 = dt * sa
    dd = 1.0 + A1 * (C - vn)
    r = I + (1.0 - scat) * dF
    kap = dt * sa / C
    em = A1 * (C + 3.0 * vn)
    gW = W * (v2 + vn * vn)
    G1, Gr, Ge = (gW / dd).sum(0), (gW * r / dd).sum(0), (gW * em / dd).sum(0)
    S0, S1 = Gr / (1.0 + kap * G1), Ge / (1.0 + kap * G1)
    W1, V1 = (W / dd).sum(0), (W * vn / dd).sum(0)
    J0 = (W * r / dd).sum(0) - kap * S0 * W1
    omJ1 = (W * (1.0 - 4.0 * A1 * vn) / dd).sum(0) + kap * S1 * W1
    H0, H1 = (W * vn * r / dd).sum(0) - kap * S0 * V1, (W * vn * em / dd).sum(0) - kap * S1 * V1
    kv = rho * (1.0 / (5.0 / 3.0 - 1.0))
    T1 = T
    if not p["hold"]:
        beta = P * C * (1.0 - v2 / C ** 2) * sa
        c0 = dt * (2.0 * FOURPI * P * sa * (H0 - S0 / C) - FOURPI * beta * J0)
        c4 = dt * (2.0 * P * sa * (H1 - S1 / C) + beta * omJ1)
        for _ in range(14):
            fn = c4 * T1 ** 4 + kv * (T1 - T) + c0
            new = T1 - fn / (4.0 * c4 * T1 ** 3 + kv)
            T1 = torch.where(new > 0, new, 0.5 * T1)
    th = T1 ** 4 / FOURPI
    I1 = (r + em * th - kap * (S0 + S1 * th)) / dd
    del dd, r, em, gW
    # scattering (sec. 4.4)
    r5 = I1 + scat * dF
    a1 = dt * ss
    ap = 1.0 + a1 * (C - vn)
    b = -a1 * C + 2.0 * a1 * vn - a1 * (v2 + vn * vn) / C
    c = -3.0 * a1 * vn
    wa = W / ap
    m11 = (W * (1.0 + a1 * vn - a1 * (v2 + vn * vn) / C) / ap).sum(0)      # 1 + sum W b / a'
    m12, m21, m22 = (wa * b * c).sum(0), wa.sum(0), 1.0 + (wa * c).sum(0)
    Br, Ar = (wa * b * r5).sum(0), (wa * r5).sum(0)
    det = m11 * m22 - m12 * m21
    s1, s2 = (Br * m22 - m12 * Ar) / det, (m11 * Ar - m21 * Br) / det
    I2 = (r5 - s1 - c * s2) / ap
    wn = wt * nt.T
    pre = wn @ (I + dF)
    Wm = torch.stack([wt, *wn, *(wn[d] * nt[:, d] for d in range(3)), wn[0] * nt[:, 1], wn[0] * nt[:, 2], wn[1] * nt[:, 2]])
    new_mom = FOURPI * (Wm @ I2)
    dM = -P / C * (new_mom[1:4] - FOURPI * pre)
    dE = kv * (T1 - T) + ((rho * v + dM).square() - (rho * v).square()).sum(0) / (2.0 * rho)
    return I2, new_mom, T1, dE, dM


def _moments64(I, nt, wt):
    wn = wt * nt.T
    Wm = torch.stack([wt, *wn, *(wn[d] * nt[:, d] for d in range(3)), wn[0] * nt[:, 1], wn[0] * nt[:, 2], wn[1] * nt[:, 2]])
    return FOURPI * (Wm @ I)


def _solve64(p, steps, fields=None, I=None):
    dev = p["rho"].device
    nt, wt = torch.tensor(p["n"], device=dev), torch.tensor(p["w"], device=dev)
    I = p["I"] if I is None else I
    mom, T = _moments64(I, nt, wt), p["T"]
    for _ in range(steps):
        I, mom, T, dE, dM = _step64(p, I, mom, T, fields or p, nt, wt)
    return I, mom, T, dE, dM


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" and case["count"] * case["steps"] > 3000:
        return None                  # thousands of small problems in turn: minutes
    if kind in ("batch", "serve"):
        got = []
        for c, s in _members(case, seed):
            p = _problem(c, s)
            if kind == "serve":      # a request starts from the isotropic equilibrium of its temperature
                p["I"] = (p["T"] ** 4 / FOURPI).expand(p["M"], p["N"])
            got.append(_solve64(p, case["steps"])[1])
        if kind == "serve":
            return [[m[0], m[1:4], m[4:10]] for m in got]
        return dict(E=torch.cat([m[0] for m in got]), F=torch.cat([m[1:4].reshape(-1) for m in got]),
                    P=torch.cat([m[4:10].reshape(-1) for m in got]))
    p = _problem(case, seed)
    I, mom, T, dE, dM = _solve64(p, case["steps"])
    if kind in ("gas", "coupled"):
        return dict(dE=dE, dM=dM if kind == "coupled" else dM.reshape(-1), T=T)
    out = dict(E=mom[0], F=mom[1:4].reshape(-1), P=mom[4:10].reshape(-1), T=T)
    if kind == "noalloc":
        out.update(dE=dE, dM=dM.reshape(-1))
        M, N, Q = p["M"], p["N"], (p["M"] + 3) // 4
        Iq = torch.zeros(4 * Q, N, dtype=torch.float64, device=I.device)
        Iq[:M] = I
        I = Iq.reshape(Q, 4, N).permute(0, 2, 1).reshape(-1)
    out["I"] = I
    return out

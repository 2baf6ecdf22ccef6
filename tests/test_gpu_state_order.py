"""Saved states of contexts that store their angles as opposite pairs: the file holds
the caller's order for every size of set, saving leaves the context as it was
(between steps of a graph, and as a member of a batch), and a loaded context goes
on bitwise."""
import numpy as np
import pytest
import torch

import paper_1403_6126_gb300 as rt

from _helpers import gpu_context
from test_gpu_pairs import C, I, P, V, _problem, _set

pytestmark = pytest.mark.gpu

OPEN = ((I, C), (V, V), (P, P))


def _context(name, shape, stream):
    n, w = _set(name)
    n, w = np.ascontiguousarray(n), np.ascontiguousarray(w)
    wl = _problem(shape, (1.0, 0.5, 0.3), OPEN, "no")
    ctx = gpu_context(wl, n, w, "fp32", stream=stream)
    ctx.set_intensity(np.random.default_rng(2).random((len(w), int(np.prod(shape)))))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    return ctx, len(w), int(np.prod(shape))


@pytest.mark.parametrize("name,shape", [
    ("s8 shuffled", (3, 7, 13)), ("s8", (1, 40, 33)), ("s2", (1, 1 + 2, 43)), ("two pairs", (2, 3, 5)), ("s6 shuffled", (12, 20, 31))])
def test_state_goes_out_and_in(name, shape):
    stream = torch.cuda.Stream().cuda_stream
    ctx, M, N = _context(name, shape, stream)
    never, _, _ = _context(name, shape, stream)
    other, _, _ = _context(name, shape, stream)
    for c in (ctx, never):
        c.run(0.0, 3)
    buf = ctx.save_state()
    quads = np.frombuffer(buf, dtype=np.float32, offset=64 + 8 * 6 * M, count=M * N).reshape(M // 4, N, 4).transpose(0, 2, 1)
    np.testing.assert_array_equal(quads.reshape(M, N), ctx.intensity().astype(np.float32))
    other.load_state(buf)
    for c in (ctx, never, other):
        c.run(0.0, 3)
        c.sync()
    for c in (ctx, other):
        np.testing.assert_array_equal(c.intensity(), never.intensity())
        for a, b in zip(c.moments(), never.moments()):
            np.testing.assert_array_equal(a, b)
    for c in (ctx, never, other):
        c.close()


def test_saving_a_batch_member_leaves_the_batch_alone():
    stream = torch.cuda.Stream().cuda_stream
    out = []
    for save in (False, True):
        members = [_context("s4", (1, 20, 33), stream)[0], _context("s6 shuffled", (5, 9, 8), stream)[0]]
        b = rt.rt_batch_create(stream)
        for c in members:
            rt.rt_batch_add(b, c.ctx)
        for _ in range(2):
            rt.rt_batch_step(b, 3)
            if save:
                for c in members:
                    c.save_state()
        out.append([c.intensity() for c in members])
        rt.rt_batch_destroy(b)
        for c in members:
            c.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)

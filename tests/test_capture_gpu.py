"""A user's CUDA graph of the library's calls: force and kdk_step captured on the
context's stream (boxes small enough for programmatic serialisation, and the forms of
the context), one box after a kernel of the user's and two boxes on a fork; every
replay gives the bits of the same calls made directly.
"""
import numpy as np
import pytest

from inputs import C1
from inputs.workloads import Level, PM3Spec
from inputs.zeldovich import random_ios

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2512_12629_gb300 import cube2  # noqa: E402

FORMS = {
    "one-level": dict(levels=(Level(64, 2.0),)),
    "two-level": dict(levels=(Level(16, 3.5), Level(64, 2.0))),
    "tsc": dict(levels=(Level(64, 2.0),), assign_order=3),
    "third-level": dict(levels=(Level(16, 3.5), Level(64, 2.0)), pm3=PM3Spec(tile=8, refine=2, beta=2.0, rho_min=20, max_tiles=64)),
    "long-streams": dict(levels=(Level(64, 2.0),)),
}
A = (0.5, 0.501, 0.502)


def _box(form, stream, seed=1):
    n_part = 70000 if form == "long-streams" else 20000
    w = C1.with_(name="capture", n_ios=32, box=32.0, b_pp=0.1, **FORMS[form])
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part), stream)
    for l in range(len(w.levels)):
        ctx.set_green(l)
    if form == "third-level":
        ctx.set_green(cube2.LEVEL_PM3)
    return ctx, cube2.IOSState.from_numpy(random_ios(n_part, 32, 32.0, seed=seed, clustered=0.3))


def _restore(p, q):
    for a, b in zip(_arrays(p), _arrays(q)):
        a.copy_(b)


def _arrays(p):
    return p.off, p.count, p.start, p.vel, p.acc


def _equal(p, q, exact=True):
    for a, b in zip(_arrays(p), _arrays(q)):
        assert torch.equal(a, b) if exact else (a.float() - b.float()).abs().max() <= 1e-5 * b.float().abs().max()


@pytest.mark.parametrize("form", FORMS)
def test_force_and_steps(form):
    s = torch.cuda.Stream()
    steps = [] if form == "tsc" else list(zip(A, A[1:]))   # its float atomics' order varies, and a step rounds positions
    with torch.cuda.stream(s):
        ctx, p = _box(form, s)
        first = p.clone()
        ctx.force(p)
        for a0, a1 in steps:
            ctx.kdk_step(p, a0, a1)
        want = p.clone()
        vel = first.vel.clone()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            p.vel.copy_(vel)            # a kernel of the user's in front
            ctx.force(p)
            for a0, a1 in steps:
                ctx.kdk_step(p, a0, a1)
        for _ in range(3):
            _restore(p, first)
            graph.replay()
            s.synchronize()
            _equal(p, want, form != "tsc")
        ctx.check()
    ctx.close()


def test_two_boxes_on_a_fork():
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        (c, p), (d, q) = _box("one-level", s, 1), _box("two-level", t, 2)
        torch.cuda.synchronize()
        first = p.clone(), q.clone()
        c.force(p)
        c.kdk_step(p, A[0], A[1])
        s.synchronize()
        with torch.cuda.stream(t):
            d.force(q)
            d.kdk_step(q, A[0], A[1])
        t.synchronize()
        want = p.clone(), q.clone()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            t.wait_stream(s)
            c.force(p)
            with torch.cuda.stream(t):
                d.force(q)
                d.kdk_step(q, A[0], A[1])
            c.kdk_step(p, A[0], A[1])
            s.wait_stream(t)
        for _ in range(3):
            _restore(p, first[0])
            _restore(q, first[1])
            graph.replay()
            torch.cuda.synchronize()
            _equal(p, want[0])
            _equal(q, want[1])
        c.check()
    c.close()
    d.close()

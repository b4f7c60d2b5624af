"""The PP kernels' source streams where they can go wrong: boxes of a few cells
(wrapped cells on both sides of a warp's block), warps of 1 to 33 targets, empty
regions wide enough for the per-lane walk, dense clumps (every pair evaluated)
with close and coincident pairs, and a softening beyond half the range; against
the FP64 oracle.

Tolerance, as for the PP force elsewhere: FP32 rounding of a sum of pair terms,
each at most the pair scale V_p / (4 pi b_cut^2), plus a term relative to the
particle's own force: |F_gpu - F_or| <= 1e-5 (scale + |F_or|).
"""
import numpy as np
import pytest

from inputs import C1
from inputs.workloads import Level
from inputs.zeldovich import ios_from_positions

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import adjoint as oadj  # noqa: E402
from oracle import kdk as okdk  # noqa: E402
from oracle import mesh as omesh  # noqa: E402
from oracle import pp as opp  # noqa: E402
from paper_2512_12629_gb300 import cube2  # noqa: E402


def _box(n, mesh, beta, b_pp):
    return C1.with_(name=f"pp-{n}", n_ios=n, box=float(n), levels=(Level(mesh, beta),), b_pp=b_pp)


def _case(name):
    rng = np.random.default_rng(7)
    if name == "four-cells":       # a warp's block and its neighbours are more cells than the box has
        w, x = _box(4, 8, 2.0, 0.1), rng.uniform(0, 4, (3, 300))
    elif name == "six-cells":
        w, x = _box(6, 12, 2.0, 0.1), np.concatenate([rng.uniform(0, 6, (3, 400)), 0.3 * rng.normal(size=(3, 200))], 1) % 6
    elif name == "wide":           # 32 targets of a pencil span more cells than a stream may
        w, x = _box(96, 96, 1.0, 0.1), np.concatenate([rng.uniform(0, 96, (3, 300)),
                                                       np.stack([rng.uniform(0, 96, 400), rng.uniform(0, 2, 400),
                                                                 rng.uniform(94, 96, 400)])], 1)
    elif name == "clump":          # every pair evaluated; many pairs closer than b_pp; coincident particles
        x = 8 + 0.25 * rng.normal(size=(3, 3000))
        x[:, 100:110] = x[:, 200:210]
        w, x = _box(16, 32, 2.0, 0.1), x
    elif name == "soft":           # b_pp beyond half the range
        w, x = _box(8, 16, 2.0, 0.7), 4 + 0.4 * rng.normal(size=(3, 900))
    else:                          # one cell of k particles
        w, x = _box(8, 16, 2.0, 0.1), 3 + rng.uniform(0, 1, (3, int(name)))
    st = ios_from_positions(x, np.zeros_like(x), w.n_ios, w.box)
    return w, st


NAMES = ["four-cells", "six-cells", "wide", "clump", "soft", "1", "31", "32", "33", "63", "65"]


@pytest.mark.parametrize("name", NAMES)
def test_pp_force(name):
    w, st = _case(name)
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    p = cube2.IOSState.from_numpy(st)
    ctx.pp_force(p)
    ctx.check()
    b_pp, b_cut = okdk.pp_params(w)
    ref = opp.pp_force(st["off"], st["count"], st["start"], w.n_ios, w.box, b_pp, b_cut)
    scale = w.box ** 3 / n_part / (4 * np.pi * b_cut ** 2)
    err = np.linalg.norm(p.acc.cpu().numpy().astype(np.float64) - ref, axis=0)
    bound = 1e-5 * (scale + np.linalg.norm(ref, axis=0))
    assert np.all(err <= bound), (err / bound).max()
    first = p.acc.clone()
    ctx.pp_count(True)                        # the counting kernel: the same forces, every pair once
    ctx.pp_force(p)
    pairs, _ = ctx.pp_stats()
    assert torch.equal(p.acc, first)
    x = omesh.positions(st["off"], st["count"], w.n_ios, w.box)
    want = oadj._pair_search(x, w.box, b_cut)[0].size
    assert abs(pairs - want) <= max(2, 1e-4 * want)
    ctx.close()


@pytest.mark.parametrize("name", ["four-cells", "six-cells", "clump", "33"])
def test_force_vjp(name):
    w, st = _case(name)
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    ctx.set_green(0)
    ctx.adjoint_init()
    p = cube2.IOSState.from_numpy(st)
    v = np.random.default_rng(1).normal(size=(3, n_part))
    got = ctx.force_vjp(p, torch.from_numpy(v.astype(np.float32)).cuda()).cpu().numpy().astype(np.float64)
    ctx.check()
    v = v.astype(np.float32).astype(np.float64)
    x = omesh.positions(st["off"], st["count"], w.n_ios, w.box)
    ref = oadj.pm_vjp_level(x, v, w.box, w.levels[0].n_mesh, n_part, omesh.green_tables(w)[0])
    b_pp, b_cut = okdk.pp_params(w)
    ref += oadj.pp_vjp_cells(st["off"], st["count"], st["start"], w.n_ios, w.box, b_pp, b_cut, v)
    err = np.linalg.norm(got - ref, axis=0)
    rel = err / np.maximum(np.linalg.norm(ref, axis=0), 1e-3 * np.sqrt(np.mean((ref ** 2).sum(0))))
    assert np.median(rel) <= 1e-5 and np.quantile(rel, 0.999) <= 1e-3, (np.median(rel), rel.max())
    ctx.close()

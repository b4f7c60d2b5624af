"""PP where the paths of the source streams change: boxes in which as many targets have
long streams as are still split between warps, and more (each stream then stays with its
warp); boxes dense throughout; warps wider than a stream may be, which walk each lane's
own cells, beside ones that are just not.  Force and adjoint product against the FP64 oracle, and the
persistent kernel bit for bit against the box's own launches.

Tolerances as in the other PP tests: |F_gpu - F_or| <= 1e-5 (scale + |F_or|) with the
pair scale V_p / (4 pi b_cut^2); the product's median 1e-5 and 99.9th percentile 1e-3
relative.
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


def _case(name):
    rng = np.random.default_rng(29)
    if name == "wide":       # 256 cells a side: pencils whose particles lie at both ends, 251, 252 and 253 cells apart
        n, mesh = 256, Level(128, 0.5)
        x = rng.uniform(0, 256, (3, 600))
        for k, gap in enumerate((250, 251, 252, 255)):
            x[0, 40 * k:40 * k + 20] = 0.5 + 0.2 * rng.normal(size=20) % 0.5
            x[0, 40 * k + 20:40 * k + 40] = gap + rng.uniform(0, 1, 20)
            x[1:, 40 * k:40 * k + 40] = np.array([[10.0], [20.0 * k + 2]]) + rng.uniform(0, 1, (2, 40))
    elif name == "even":     # eight a cell: between the warps that evaluate every pair and those that test first
        n, mesh = 16, Level(32, 2.0)
        x = np.concatenate([rng.uniform(0, 16, (3, 33000)), 8 + rng.normal(size=(3, 1000))], 1) % 16
    else:                    # 16^3 cells, evenly: every stream is long
        n, mesh = 16, Level(32, 2.0)
        x = rng.uniform(0, 16, (3, int(name)))
    w = C1.with_(name=f"crowd-{name}", n_ios=n, box=float(n), levels=(mesh,), b_pp=0.1)
    return w, ios_from_positions(x, np.zeros_like(x), n, w.box)


NAMES = ["90000", "100000", "even", "wide"]


@pytest.mark.parametrize("name", NAMES)
def test_force(name):
    w, st = _case(name)
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    p = cube2.IOSState.from_numpy(st)
    ctx.pp_force(p)
    ctx.check()
    b_pp, b_cut = okdk.pp_params(w)
    some = np.arange(0, n_part, max(1, n_part // 3000))
    ref = opp.pp_force_at_many(st["off"], st["count"], st["start"], w.n_ios, w.box, b_pp, b_cut, some)
    scale = w.box ** 3 / n_part / (4 * np.pi * b_cut ** 2)
    err = np.linalg.norm(p.acc.cpu().numpy()[:, some].astype(np.float64) - ref, axis=0)
    bound = 1e-5 * (scale + np.linalg.norm(ref, axis=0))
    assert np.all(err <= bound), (err / bound).max()
    first = p.acc.clone()
    ctx.pp_count(True)
    ctx.pp_force(p)
    assert torch.equal(p.acc, first)
    if name == "wide":
        lane = ctx.pp_stats_paths()[2:]
        assert lane[1] > 0                    # some warps walked
    ctx.close()


@pytest.mark.parametrize("name", NAMES[1:2] + NAMES[3:])
def test_force_vjp(name):
    w, st = _case(name)
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    ctx.set_green(0)
    ctx.adjoint_init()
    p = cube2.IOSState.from_numpy(st)
    v = np.random.default_rng(1).normal(size=(3, n_part)).astype(np.float32)
    got = ctx.force_vjp(p, torch.from_numpy(v).cuda()).cpu().numpy().astype(np.float64)
    ctx.check()
    v = v.astype(np.float64)
    x = omesh.positions(st["off"], st["count"], w.n_ios, w.box)
    ref = oadj.pm_vjp_level(x, v, w.box, w.levels[0].n_mesh, n_part, omesh.green_tables(w)[0])
    b_pp, b_cut = okdk.pp_params(w)
    ref += oadj.pp_vjp_cells(st["off"], st["count"], st["start"], w.n_ios, w.box, b_pp, b_cut, v)
    err = np.linalg.norm(got - ref, axis=0)
    rel = err / np.maximum(np.linalg.norm(ref, axis=0), 1e-3 * np.sqrt(np.mean((ref ** 2).sum(0))))
    assert np.median(rel) <= 1e-5 and np.quantile(rel, 0.999) <= 1e-3, (np.median(rel), rel.max())
    ctx.close()


@pytest.mark.parametrize("name", NAMES)
def test_persistent_kernel_gives_the_same_bits(name):
    w, st = _case(name)
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    ctx.set_green(0)
    p = cube2.IOSState.from_numpy(st)
    ctx.force(p)
    want = p.clone()
    ctx.kdk_step(want, 0.5, 0.50001)
    ens = cube2.Ensemble([ctx], [p], np.array([[0.5, 0.50001]]), opts=cube2.ensemble_opts(n_streams=1, persistent_pp=True))
    ens.launch()
    ens.check()
    assert torch.equal(p.acc, want.acc) and torch.equal(p.vel, want.vel) and torch.equal(p.off, want.off)
    ens.close()
    ctx.close()

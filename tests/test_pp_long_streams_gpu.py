"""Warps whose source stream is shared by several warps (boxes of 65536 particles
or more, streams of more than 512 sources): a clump across the box's corner in an
even background, so that long streams have wrapped cells and every length around
the line occurs; the force and the adjoint's product against the FP64 oracle, the
pair counts, and the ensemble's persistent kernel, which works on the parts one
after another, bit for bit against the box's own launches.

Tolerances as in the other PP tests: |F_gpu - F_or| <= 1e-5 (scale + |F_or|) with
the pair scale V_p / (4 pi b_cut^2); the product's median 1e-5 and 99.9th
percentile 1e-3 relative.
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

N_IOS = 32


@pytest.fixture(scope="module")
def case():
    rng = np.random.default_rng(17)
    x = np.concatenate([rng.uniform(0, N_IOS, (3, 62537)), 0.5 * rng.normal(size=(3, 2500)),
                        16 + 1.2 * rng.normal(size=(3, 500))], axis=1) % N_IOS
    w = C1.with_(name="pp-long", n_ios=N_IOS, box=float(N_IOS), levels=(Level(2 * N_IOS, 2.0),), b_pp=0.1)
    return w, ios_from_positions(x, np.zeros_like(x), N_IOS, w.box)


@pytest.mark.parametrize("drop", [0, 1])   # 65537 and 65536 particles: at the line
def test_force(case, drop):
    w, st = case
    n_part = int(st["count"].sum())
    if drop:
        x = omesh.positions(st["off"], st["count"], N_IOS, w.box)[:, drop:]
        st, n_part = ios_from_positions(x, np.zeros_like(x), N_IOS, w.box), n_part - drop
    assert n_part == 65537 - drop
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    p = cube2.IOSState.from_numpy(st)
    ctx.pp_force(p)
    ctx.check()
    b_pp, b_cut = okdk.pp_params(w)
    ref = opp.pp_force(st["off"], st["count"], st["start"], N_IOS, w.box, b_pp, b_cut)
    scale = w.box ** 3 / n_part / (4 * np.pi * b_cut ** 2)
    err = np.linalg.norm(p.acc.cpu().numpy().astype(np.float64) - ref, axis=0)
    bound = 1e-5 * (scale + np.linalg.norm(ref, axis=0))
    assert np.all(err <= bound), (err / bound).max()
    first = p.acc.clone()
    ctx.pp_count(True)
    ctx.pp_force(p)
    assert torch.equal(p.acc, first)
    x = omesh.positions(st["off"], st["count"], N_IOS, w.box)
    want = oadj._pair_search(x, w.box, b_cut)[0].size
    assert abs(ctx.pp_stats()[0] - want) <= max(2, 1e-4 * want)
    ctx.close()


def test_force_vjp(case):
    w, st = case
    n_part = int(st["count"].sum())
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=n_part))
    ctx.set_green(0)
    ctx.adjoint_init()
    p = cube2.IOSState.from_numpy(st)
    v = np.random.default_rng(1).normal(size=(3, n_part)).astype(np.float32)
    got = ctx.force_vjp(p, torch.from_numpy(v).cuda()).cpu().numpy().astype(np.float64)
    ctx.check()
    v = v.astype(np.float64)
    x = omesh.positions(st["off"], st["count"], N_IOS, w.box)
    ref = oadj.pm_vjp_level(x, v, w.box, 2 * N_IOS, n_part, omesh.green_tables(w)[0])
    b_pp, b_cut = okdk.pp_params(w)
    ref += oadj.pp_vjp_cells(st["off"], st["count"], st["start"], N_IOS, w.box, b_pp, b_cut, v)
    err = np.linalg.norm(got - ref, axis=0)
    rel = err / np.maximum(np.linalg.norm(ref, axis=0), 1e-3 * np.sqrt(np.mean((ref ** 2).sum(0))))
    assert np.median(rel) <= 1e-5 and np.quantile(rel, 0.999) <= 1e-3, (np.median(rel), rel.max())
    ctx.close()


def test_persistent_kernel_gives_the_same_bits(case):
    w, st = case
    n_part = int(st["count"].sum())
    ctxs = [cube2.init_mesh(cube2.make_config(w, n_particles=n_part)) for _ in range(2)]
    for c in ctxs:
        c.set_green(0)
    states = [cube2.IOSState.from_numpy(st) for _ in ctxs]
    for c, p in zip(ctxs, states):
        c.force(p)
    want = states[0].clone()
    ctxs[0].kdk_step(want, 0.5, 0.501)
    ens = cube2.Ensemble(ctxs, states, np.array([[0.5, 0.501]] * 2), opts=cube2.ensemble_opts(n_streams=2, persistent_pp=True))
    ens.launch()
    ens.check()
    for p in states:
        assert torch.equal(p.acc, want.acc) and torch.equal(p.vel, want.vel) and torch.equal(p.off, want.off)
    ens.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("width", [8, 16])
def test_stream_width_option_leaves_the_bits(width):
    # thin boxes, whose warps span many cells: the option once moved them to the per-lane walk
    rng = np.random.default_rng(3)
    w = C1.with_(name="thin", n_ios=N_IOS, box=float(N_IOS), levels=(Level(N_IOS, 1.0),), b_pp=0.1)
    x = rng.uniform(0, N_IOS, (3, 9000))
    st = ios_from_positions(x, np.zeros_like(x), N_IOS, w.box)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=9000))
    ctx.set_green(0)
    p = cube2.IOSState.from_numpy(st)
    ctx.force(p)
    want = p.clone()
    ctx.kdk_step(want, 0.5, 0.501)
    ens = cube2.Ensemble([ctx], [p], np.array([[0.5, 0.501]]),
                         opts=cube2.ensemble_opts(n_streams=1, persistent_pp=True, pp_wmax=width))
    ens.launch()
    ens.check()
    assert torch.equal(p.acc, want.acc) and torch.equal(p.vel, want.vel) and torch.equal(p.off, want.off)
    ens.close()
    ctx.close()

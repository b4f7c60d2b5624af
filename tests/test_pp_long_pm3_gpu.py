"""Long source streams in a third-level context (65537 particles): targets in refined
subtiles have the local range, the others the finest level's, in one warp and in one
shared stream; PP alone against the FP64 oracle with either range.

Tolerance, as in the other PP tests: |F_gpu - F_or| <= 1e-5 (scale + |F_or|) with the
pair scale V_p / (4 pi b^2) of the shorter range.
"""
import numpy as np
import pytest

from inputs import C1
from inputs.workloads import Level, PM3Spec
from inputs.zeldovich import ios_from_positions

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import kdk as okdk  # noqa: E402
from oracle import pp as opp  # noqa: E402
from paper_2512_12629_gb300 import cube2  # noqa: E402

N_IOS, N_PART, TILE = 32, 65537, 8


def test_force():
    rng = np.random.default_rng(23)
    x = np.concatenate([rng.uniform(0, N_IOS, (3, N_PART - 3000)), 0.5 * rng.normal(size=(3, 2500)),
                        16 + 1.2 * rng.normal(size=(3, 500))], axis=1) % N_IOS     # both clumps on subtile corners
    w = C1.with_(name="pp-long-pm3", n_ios=N_IOS, box=float(N_IOS), levels=(Level(16, 3.5), Level(2 * N_IOS, 2.0)), b_pp=0.1,
                 pm3=PM3Spec(tile=TILE, refine=2, beta=2.0, rho_min=40, max_tiles=8))
    st = ios_from_positions(x, np.zeros_like(x), N_IOS, w.box)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=N_PART))
    p = cube2.IOSState.from_numpy(st)
    ctx.pp_force(p)
    ctx.check()
    b_pp, b_cut = okdk.pp_params(w)
    b3 = ctx.pm3_info()["b3"]
    ns = N_IOS // TILE
    cell = np.repeat(np.arange(N_IOS ** 3), st["count"])
    cz, cy, cx = cell // N_IOS ** 2, cell // N_IOS % N_IOS, cell % N_IOS
    slot = ctx.pm3_map().cpu().numpy()
    refined = slot[(cz // TILE * ns + cy // TILE) * ns + cx // TILE] >= 0
    assert 0 < refined.sum() < N_PART and (slot < 0).any()
    args = st["off"], st["count"], st["start"], N_IOS, w.box, b_pp
    ref = np.where(refined, opp.pp_force(*args, b3), opp.pp_force(*args, b_cut))
    scale = w.box ** 3 / N_PART / (4 * np.pi * b3 ** 2)
    err = np.linalg.norm(p.acc.cpu().numpy().astype(np.float64) - ref, axis=0)
    bound = 1e-5 * (scale + np.linalg.norm(ref, axis=0))
    assert np.all(err <= bound), (err / bound).max()
    first = p.acc.clone()
    ctx.pp_count(True)
    ctx.pp_force(p)
    assert torch.equal(p.acc, first)
    ctx.close()

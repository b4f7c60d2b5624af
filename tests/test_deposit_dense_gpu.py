"""The CIC deposit in evenly dense boxes, where bricks go from one division of their
particles to the other: lanes on single particles and on runs of four, coarse blocks by
threads and by warps (128 particles, four times the average of those, 4096), with and without
clumps, whole and partial bricks; accumulators and FP32 grids against the oracle's
integers, bit for bit.
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

from oracle import mesh as omesh  # noqa: E402
from paper_2512_12629_gb300 import cube2  # noqa: E402


@pytest.mark.parametrize("n,meshes,per_cell,clump", [
    (16, (8, 32), 2.9, 0), (16, (8, 32), 3.2, 0), (16, (8, 16), 13, 0), (16, (8, 32), 20, 3000), (24, (12, 24), 14, 900),
    (12, (12, 48), 30, 2000), (24, (12, 48), 5, 400), (16, (8,), 500, 0), (16, (8,), 530, 20000), (16, (32,), 40, 0)])
def test_deposit_is_exact(n, meshes, per_cell, clump):
    rng = np.random.default_rng(n + clump)
    x = np.concatenate([rng.uniform(0, n, (3, int(per_cell * n ** 3))), (5.0 + rng.uniform(-1, 1, (3, clump)))], axis=1)
    st = ios_from_positions(x % n, np.zeros_like(x), n, float(n))
    count = int(st["count"].sum())
    levels = tuple(Level(m, 0.4 * m / n) for m in meshes)
    ctx = cube2.init_mesh(cube2.make_config(C1.with_(name="dense", n_ios=n, box=float(n), levels=levels, b_pp=0.05),
                                            n_particles=count))
    p = cube2.IOSState.from_numpy(st)
    ctx.deposit(-1, p)
    for l, m in enumerate(meshes):
        want = omesh.deposit_u64(st["off"], st["count"], n, m)
        d32 = ctx.get_density(l).cpu().numpy()
        assert np.array_equal(d32.view(np.uint32), omesh.density_fp32(want, count).view(np.uint32))
        assert np.array_equal(ctx.deposit_u64(l, p).cpu().numpy().view(np.uint64), want)
    ctx.check()
    ctx.close()

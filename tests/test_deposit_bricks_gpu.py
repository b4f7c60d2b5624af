"""The CIC deposit's bricks where they can go wrong: meshes of half, one, two and
four times the IOS resolution, partial bricks, boxes smaller than a brick, runs of
particles long enough for a warp, for chunked lanes and for the overflow watch;
accumulators and FP32 grids against the oracle's integers, bit for bit.
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


def _state(n, dense, seed):
    """1500 even particles and `dense` ones in two neighbouring cells of a corner of the box."""
    rng = np.random.default_rng(seed)
    x = np.concatenate([rng.uniform(0, n, (3, 1500)), rng.uniform(0, 1, (3, dense)) * [[2.0], [1.0], [1.0]] - 1.0], axis=1)
    return ios_from_positions(x % n, np.zeros_like(x), n, float(n))


@pytest.mark.parametrize("dense", [0, 95, 97, 5000, 70000])
@pytest.mark.parametrize("n,meshes", [(4, (8,)), (6, (12,)), (12, (12, 24)), (16, (8, 32)), (24, (12, 96)), (16, (8,)),
                                      (24, (24,))])
def test_deposit_is_exact(n, meshes, dense):
    st = _state(n, dense, n + dense)
    count = int(st["count"].sum())
    levels = tuple(Level(m, 0.4 * m / n) for m in meshes)   # softening within the IOS cell on every level
    w = C1.with_(name="bricks", n_ios=n, box=float(n), levels=levels, b_pp=0.05)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=count))
    p = cube2.IOSState.from_numpy(st)
    want = [omesh.deposit_u64(st["off"], st["count"], n, m) for m in meshes]
    for l, acc in enumerate(want):
        assert np.array_equal(ctx.deposit_u64(l, p).cpu().numpy().view(np.uint64), acc)
    for level in [-1] + list(range(len(meshes))):
        ctx.deposit(level, p)
        for l, acc in enumerate(want):
            if level in (-1, l):
                d32 = ctx.get_density(l).cpu().numpy()
                assert np.array_equal(d32.view(np.uint32), omesh.density_fp32(acc, count).view(np.uint32))
    ctx.check()
    ctx.close()


@pytest.mark.parametrize("over", [0, 1])
def test_coarse_overflow(over):
    """65535 particles at a coarse mesh-cell centre fit in 64 bits, one more sets the capacity word."""
    n, k = 16, 65535 + over
    x = np.full((3, k), 5.0)      # coarse cell 2's centre: IOS cell boundary 5
    st = ios_from_positions(x, np.zeros_like(x), n, float(n))
    w = C1.with_(name="over", n_ios=n, box=float(n), levels=(Level(8, 0.2),), b_pp=0.05)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=k))
    ctx.deposit(0, cube2.IOSState.from_numpy(st))
    if over:
        with pytest.raises(cube2.Cube2Error) as e:
            ctx.check()
        assert e.value.code == cube2.ERR_CAPACITY
    else:
        ctx.check()
    ctx.close()

"""The re-bin and the placement around the sizes at which a cell's particles change
hands: ranked in the gather up to 160, one warp up to 256, one CTA above (8192 at a
time); cells at the start and the end of the list, particle counts around a warp.
The orders are those of a stable sort by cell, exactly; the FP16 scales are the
cells' largest components, exactly.
"""
import numpy as np
import pytest

from inputs import C1
from inputs.workloads import Level

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2512_12629_gb300 import cube2  # noqa: E402


@pytest.mark.parametrize("sizes,rest,fp16", [((1, 2), 28, False), ((1, 2), 30, True), ((159, 160), 1000, True),
                                             ((161, 256), 999, False), ((257, 255), 1, False),
                                             ((8192, 8193), 5000, True), ((1025, 512), 0, False)])
def test_order_is_the_stable_one(sizes, rest, fp16):
    n = 6                                    # 216 cells
    rng = np.random.default_rng(sum(sizes) + rest)
    cells = np.concatenate([np.zeros(sizes[0], int), np.full(sizes[1], n ** 3 - 1), rng.integers(0, n ** 3, rest)])
    rng.shuffle(cells)
    count = cells.size
    off = rng.integers(0, 65536, (3, count))
    xyz = np.stack([cells % n, cells // n % n, cells // n ** 2])
    pos = xyz + off / 65536.0                # exact in FP64: s_ios is 1
    mom = rng.normal(size=(3, count)).astype(np.float32)
    order = np.argsort(cells, kind="stable")
    w = C1.with_(name="ranks", n_ios=n, box=float(n), levels=(Level(2 * n, 0.8),), b_pp=0.05)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=count))
    p, perm = cube2.ios_from_positions(ctx, torch.tensor(pos, device="cuda"), torch.tensor(mom, device="cuda"))
    assert np.array_equal(perm.cpu().numpy(), order)
    got = p.to_numpy()
    assert np.array_equal(got["vel"], mom[:, order])
    assert np.array_equal(got["count"].ravel(), np.bincount(cells, minlength=n ** 3))
    assert np.array_equal(got["off"].astype(int), off[:, order])
    if fp16:
        ctx.close()
        config = cube2.make_config(w, n_particles=count)
        config.vel_fp16 = 1
        ctx = cube2.init_mesh(config)
        ctx.vel_encode(p, p.vel)
        scale = np.zeros(n ** 3, np.float32)
        np.maximum.at(scale, cells, np.abs(mom).max(axis=0))
        assert np.array_equal(p.vscale.cpu().numpy().ravel(), scale)
    ctx.set_green(0)
    ctx.force(p)
    before = p.off.clone()
    ctx.kdk_step(p, 0.5, 0.5 + 1e-12)        # moves nobody: the order stays
    assert torch.equal(p.off, before)
    ctx.check()
    ctx.close()


@pytest.mark.parametrize("box", [6.0, 7.3, 6.0e-7, 6.0e31])
def test_positions_round_as_fp64_division_does(box):
    # the placement's integer quotient: halves and their neighbours, whole values,
    # other periods and signs, zeros, the smallest values and those past 2^31
    n = 6
    s_ios = box / n
    rng = np.random.default_rng(11)
    u = np.concatenate([rng.integers(-2 ** 30, 2 ** 30, 4000) + 0.5, rng.integers(0, n * 65536, 4000) + 0.5,
                        rng.integers(-10 ** 6, 10 ** 6, 4000), rng.uniform(-2e6, 2e6, 20000), rng.uniform(-2e12, 2e12, 4000),
                        rng.choice([-1.0, 1.0], 4000) * 10.0 ** rng.uniform(-300, 9, 4000), np.arange(-8, 8) * 0.25])
    x = u * (s_ios / 65536.0)
    x = np.concatenate([x, np.nextafter(x, np.inf), np.nextafter(x, -np.inf), x + 2.0 ** -21 * s_ios, [0.0, -0.0, 5e-324]])
    x = x[:3 * (x.size // 3)].reshape(3, -1)
    X = np.rint(x / s_ios * 65536.0).astype(np.int64) % (n * 65536)
    cells = (X >> 16)[0] + n * ((X >> 16)[1] + n * (X >> 16)[2])
    order = np.argsort(cells, kind="stable")
    w = C1.with_(name="round", n_ios=n, box=box, levels=(Level(2 * n, 0.8),), b_pp=0.05 * s_ios)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=x.shape[1]))
    p, perm = cube2.ios_from_positions(ctx, torch.tensor(x, device="cuda"))
    assert np.array_equal(perm.cpu().numpy(), order)
    assert np.array_equal(p.off.cpu().numpy().view(np.uint16).astype(int), (X & 0xffff)[:, order])
    ctx.check()
    bad = torch.tensor(x, device="cuda")
    bad[1, 7] = float("inf")
    cube2.ios_from_positions(ctx, bad)
    with pytest.raises(cube2.Cube2Error):
        ctx.check()
    ctx.close()

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

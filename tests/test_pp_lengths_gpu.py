"""PP with softenings and ranges below the particles' resolution of 2^-16 IOS cells.
Two particles are at no distance or at 2^-16 cells at least, so every softening below
that gives the bits of every other, a range below it no force at all, and each warp's
path (every pair, queues, the per-lane walk) leaves the target itself out.
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

from paper_2512_12629_gb300 import cube2  # noqa: E402


def _state(name):
    rng = np.random.default_rng(5)
    if name == "clump":
        n, x = 16, 8 + 0.25 * rng.normal(size=(3, 1500))
        x[:, 10:14] = x[:, 20:24]
    elif name == "even":
        n, x = 16, rng.uniform(0, 16, (3, 4096))
    else:                                    # "wide": the per-lane walk
        n, x = 96, rng.uniform(0, 96, (3, 300))
        x[:, :100] = (x[:, 100:200] + 0.3) % 96
    return n, ios_from_positions(x, np.zeros_like(x), n, float(n))


def _forces(n, st, beta, b_pp):
    w = C1.with_(name="lengths", n_ios=n, box=float(n), levels=(Level(n, beta),), b_pp=b_pp)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=int(st["count"].sum())))
    p = cube2.IOSState.from_numpy(st)
    ctx.pp_force(p)
    ctx.check()
    ctx.close()
    return p.acc


@pytest.mark.parametrize("b_pp", [1e-30, 1e-23, 1e-12, 2.0 ** -17])
@pytest.mark.parametrize("name", ["clump", "even", "wide"])
def test_softening(name, b_pp):
    n, st = _state(name)
    want = _forces(n, st, 1.0, 2.0 ** -18)
    assert want.abs().max() > 0
    assert torch.equal(_forces(n, st, 1.0, b_pp), want)


@pytest.mark.parametrize("name", ["clump", "even", "wide"])
def test_range(name):
    n, st = _state(name)
    for b_range in (1e-14, 1e-20, 2.0 ** -17):
        assert (_forces(n, st, b_range, 1e-30) == 0).all()

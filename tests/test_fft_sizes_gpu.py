"""Every mesh size the line transforms are instantiated for up to 512 (each radix
sequence, threads per line and tile shape): the forward spectrum and the Poisson
solve of a random density against numpy in FP64.

Tolerances, as elsewhere for the solve: relative L2 of the spectrum below
2e-7 log2 n, potential within 1e-5 of its largest value.
"""
import numpy as np
import pytest

from inputs import C1
from inputs.workloads import Level
from inputs.zeldovich import random_ios

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2512_12629_gb300 import cube2  # noqa: E402


@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512])
def test_forward_and_solve(n):
    ni = n if n == 12 else n // 2
    w = C1.with_(name=f"fft-{n}", n_ios=ni, box=float(ni), levels=(Level(n, 1.0 if n == 12 else 2.0),), b_pp=0.05)
    st = random_ios(4000, ni, w.box, seed=n, clustered=0.5)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=4000))
    ctx.set_green(0)
    p = cube2.IOSState.from_numpy(st)
    ctx.deposit(0, p)
    rho = ctx.get_density(0).cpu().numpy().astype(np.float64)
    ref = np.fft.rfftn(rho)
    got = ctx.debug_forward_fft(0).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 2e-7 * np.log2(n) * np.linalg.norm(ref)
    ctx.deposit(0, p)
    ctx.solve_pm(0)
    phi = ctx.get_potential(0).cpu().numpy().astype(np.float64)
    green = ctx.get_green(0).cpu().numpy().astype(np.float64) * n ** 3   # the table carries 1/n^3
    want = np.fft.irfftn(ref * green, s=(n, n, n), axes=(0, 1, 2))
    assert np.abs(phi - want).max() <= 1e-5 * np.abs(want).max()
    ctx.check()
    ctx.close()

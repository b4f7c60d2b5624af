"""The allocation-free Poisson solve at the sizes that test_zz_no_alloc leaves out,
against cube2_solve_pm on the same density and Green's table, each twice and once more
after a larger and a smaller mesh have used the fixed array.

Tolerance, as there: 1e-5 of the largest potential.
"""
import ctypes

import pytest

from inputs.workloads import Level, Workload
from inputs.zeldovich import random_ios

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2512_12629_gb300 import cube2  # noqa: E402


def _case(n):
    w = Workload(name=f"noalloc-{n}", n_p=n // 2, box=float(n // 2), n_ios=n // 2, levels=(Level(n, 2.0),), b_pp=0.1)
    st = random_ios(2000, n // 2, w.box, seed=n, clustered=0.5)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=2000))
    ctx.set_green(0)
    ctx.deposit(0, cube2.IOSState.from_numpy(st))
    rho, green = ctx.get_density(0), ctx.get_green(0)
    ctx.solve_pm(0)
    ref = ctx.get_potential(0)
    ctx.check()
    ctx.close()
    return rho, green, ref


def _check(n, case):
    rho, green, ref = case
    out = torch.full_like(rho, float("nan"))
    rc = cube2.library().cube2_solve_pm_noalloc(rho.data_ptr(), green.data_ptr(), out.data_ptr(), n,
                                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == cube2.OK
    torch.cuda.synchronize()
    assert ((out - ref).abs().max() <= 1e-5 * ref.abs().max()).item()


@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 96])
def test_solve(n):
    case = _case(n)
    for _ in range(2):
        _check(n, case)
    for other in (128, 48):
        _check(other, _case(other))
    _check(n, case)

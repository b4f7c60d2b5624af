"""The autotuner leaves the option without effect (the stream width) as it was given."""
import numpy as np
import pytest

from inputs.workloads import c4_ensemble
from inputs.zeldovich import zeldovich_ios

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2512_12629_gb300 import cube2  # noqa: E402


def test_autotuner_keeps_the_width():
    w = c4_ensemble(n_boxes=1, seed=5, n_steps=1, sizes=(16,))[0]
    st = zeldovich_ios(w)
    ctx = cube2.init_mesh(cube2.make_config(w, n_particles=int(st["count"].sum())))
    ctx.set_green(0)
    p = cube2.IOSState.from_numpy(st)
    ctx.force(p)
    a0 = 1.0 / (1.0 + w.z_init)
    best, _ = cube2.ensemble_autotune([ctx], [p], np.array([[a0, a0 + 0.01]]),
                                      start=cube2.ensemble_opts(n_streams=8, persistent_pp=True, pp_ctas_per_sm=4, pp_wmax=8),
                                      trials=1)
    assert best.pp_wmax == 8 and best.persistent_pp == 1
    ctx.check()
    ctx.close()

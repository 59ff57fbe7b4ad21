"""A shear Wiener filter whose max_iter ends within the cooling levels: not converged, with no residual measured."""
import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [64, 128, 256, 512])
def test_max_iter_within_the_cooling_levels(H):
    need_gpu()
    build.build()
    d, N, m, P = to_dev(synth.make_problem(H, seed=H, mask_frac=0.1, k0=1.0 / 32))
    r = wf.wf_solve_spin2(d, d, N, N, m, P, P, max_iter=1, allow_not_converged=True)
    assert r.status == 5 and r.resid == -1.0 and r.iters >= 64
    assert torch.isfinite(r.s).all() and float(r.s.abs().max()) > 0   # the last cooling level's map

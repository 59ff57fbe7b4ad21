"""The large-image switch at 128 x 128: "cluster" runs the kernels that "auto" runs (clusters, where they fit), no slower."""
import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


def _ms(call, mode):
    wf.wf_set_large_image_sampler(mode)
    wf.wf_set_kernel_timing(True)
    try:
        out = call()
        ms = []
        for _ in range(5):
            call()
            ms.append(wf.wf_last_kernel_ms())
        return out, sorted(ms)[2]
    finally:
        wf.wf_set_kernel_timing(False)
        wf.wf_set_large_image_sampler("auto")


@pytest.mark.parametrize("kind,count", [("sample", 1), ("sample", 40), ("solve", 1), ("shear", 1), ("shear", 30)])
def test_cluster_runs_as_auto(kind, count):
    """A sweep takes 3.8 to 5.6 us in clusters and 6 to 9 us in the global-memory kernels; the results are equal bit for bit
    (the same kernel)."""
    need_gpu()
    build.build()
    dev = to_dev(synth.make_problem(128, seed=1, mask_frac=0.1, k0=1.0 / 32))
    if kind == "sample":
        call = lambda: wf.wf_sample_ex(*dev, seed=3, n_samples=1, n_chains=count, thin=400)  # noqa: E731
    elif kind == "solve":
        call = lambda: wf.wf_solve_ex(*dev, tol=1e-5, refine=0).s  # noqa: E731
    else:
        d, N, mask, P = dev
        call = lambda: wf.wf_sample_spin2(d, d, N, N, mask, P, P, 3, 1, n_chains=count, thin=400)  # noqa: E731
    a, t_auto = _ms(call, "auto")
    b, t_cluster = _ms(call, "cluster")
    assert torch.equal(a, b)
    assert t_cluster < 1.15 * t_auto, (t_auto, t_cluster)

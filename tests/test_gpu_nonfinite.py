"""A residual that overflows FP32 ends the Wiener filter with the non-finite status, on every kernel that decides the
schedule, instead of running on to max_iter."""
import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


def _overflowing(H):
    """Finite inputs whose residual and level norms, sums of squares of 1e25, are infinite in FP32 (and not NaN: every
    mode has power)."""
    p = synth.make_problem(H, seed=H, mask_frac=0.1)
    p.Pk[0, 0] = p.Pk[0, 1]
    d, N, mask, Pk = to_dev(p)
    return d * 1e25, N, mask, Pk


@pytest.fixture(autouse=True)
def _lib():
    need_gpu()
    build.build()
    yield
    wf.wf_set_large_image_sampler("auto")


@pytest.mark.parametrize("H,mode", [(16, "auto"), (32, "auto"), (64, "auto"), (128, "auto"), (128, "global"), (256, "auto"),
                                    (256, "global"), (256, "cluster"), (512, "auto"), (512, "global"), (512, "cluster"),
                                    (1024, "auto"), (1024, "global")])
def test_filter(H, mode):
    wf.wf_set_large_image_sampler(mode)
    with pytest.raises(wf.WFError) as e:
        wf.wf_solve_ex(*_overflowing(H), refine=0, max_iter=400)
    assert e.value.status == 6


@pytest.mark.parametrize("small_path", [0, 1])
def test_batch(small_path):
    """Next to a finite image of each size class, which converges."""
    sizes = [16, 32, 64, 128, 256, 512]
    bad = [wf.BatchImage(*_overflowing(H)) for H in sizes]
    good = [wf.BatchImage(*to_dev(synth.make_problem(H, seed=H, mask_frac=0.1))) for H in sizes]
    with pytest.raises(wf.WFError) as e:
        wf.wf_batch_run([x for pair in zip(good, bad) for x in pair], max_iter=400, small_path=small_path)
    assert e.value.status == 6
    assert [x.status for x in bad] == [6] * len(sizes)
    assert [x.status for x in good] == [0] * len(sizes)
    assert all(torch.isfinite(x.out_wf).all() for x in good)

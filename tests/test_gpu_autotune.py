"""The batch autotuner leaves the options that reach no kernel of the batch as the caller gave them."""
import pytest

from gpu_common import need_gpu, to_dev
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


def test_options_without_effect_are_not_tried():
    """One 64^2 and one 512^2 image on the global-memory kernels: no clusters to share out or to shape, one large class on
    one stream, and no 16^2 image. A candidate without effect wins by noise about every other time, so five runs that tried
    them would change one of these values with near certainty."""
    need_gpu()
    build.build()
    images = [wf.BatchImage(*to_dev(synth.make_problem(H, seed=H, mask_frac=0.1))) for H in (64, 512)]
    for _ in range(5):
        chosen, ms = wf.wf_batch_autotune(images, n_samples=2, reps=1)
        assert ms > 0
        assert chosen["large_streams"] == 8 and chosen["large_cluster_rows"] == 0 and chosen["small_fields_per_cta"] == 0

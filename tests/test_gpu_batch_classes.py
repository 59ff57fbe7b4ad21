"""Large batch classes in one launch, of fewer and of more work items than CTAs: every image's result is
that of the image in a batch of its own (the same passes; the residual sums are added in another order in FP64)."""
import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,count", [(256, 28), (256, 29), (256, 70), (512, 7), (512, 8), (512, 20), (1024, 3)])
def test_images_of_a_class_equal_single_batches(H, count):
    need_gpu()
    build.build()
    pool = []
    for i in range(min(count, 6)):  # solves of different lengths
        pool.append(to_dev(synth.make_problem(H, seed=H + i, mask_frac=0.05 * i, slope=-1.0 - 0.4 * i, k0=1.0 / 32,
                                              sigma2=(0.01, 0.05 + 0.1 * i))))
    bad = [x.clone() for x in pool[0]]
    bad[0][0, 0] = float("nan")  # an image whose set-up fails takes no part
    images = [wf.BatchImage(*(bad if i == 1 else pool[i % len(pool)]), seed=3, chain=i) for i in range(count)]
    with pytest.raises(wf.WFError):
        wf.wf_batch_run(images, n_samples=2)
    assert images[1].status == 6 and len({im.iters for im in images}) > 2
    for i in sorted({0, 2, count // 2, count - 1} - {1}):
        im = images[i]
        one = wf.BatchImage(im.d, im.Ndiag, im.mask, im.Pk, seed=3, chain=i)
        wf.wf_batch_run([one], n_samples=2)
        assert im.status == 0 and one.iters == im.iters
        assert torch.equal(one.out_wf, im.out_wf) and torch.equal(one.out_samples, im.out_samples)

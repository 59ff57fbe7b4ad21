"""GPU checks of the sampler's kernel choice by chain count: the one-thread-per-row kernel (many 64 x 64 chains) and the
kernel with several threads per row, and the cluster and global-memory kernels at 256 x 256, draw the same chains."""
import pytest

from gpu_common import need_gpu, rel, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,chains", [(32, 1), (32, 67), (64, 1), (64, 760), (64, 761), (64, 1217), (128, 35), (128, 36), (128, 305), (256, 399),
                                      (256, 400), (512, 9)])
def test_chain_does_not_depend_on_the_chain_count(H, chains):
    """Chain c of a call with many chains equals the call for that chain alone. Each kernel is within 5e-7
    relative L2 of the exact chain (FP32 rounding over these sweeps), so the two agree to 2e-6."""
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H, mask_frac=0.1, block=(1, H // 4, 2, H // 3))
    dev = to_dev(p)
    many = wf.wf_sample_ex(*dev, seed=7, n_samples=2, n_chains=chains, burn_in=2, thin=3)
    for c in sorted({0, chains // 2, chains - 1}):
        one = wf.wf_sample_ex(*dev, seed=7, n_samples=2, n_chains=1, chain_offset=c, burn_in=2, thin=3)
        assert rel(many[c].cpu().numpy(), one[0].cpu().numpy()) < 2e-6, (H, chains, c)


@pytest.mark.parametrize("H,chains", [(32, 3), (64, 2), (128, 39), (128, 40), (256, 23), (256, 24), (512, 2)])
def test_shear_chain_does_not_depend_on_the_chain_count_or_path(H, chains):
    """Both kernels of the spin-2 sampler draw the same chains (2e-6: FP32 rounding of either)."""
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H, mask_frac=0.1)
    q = synth.make_problem(H, seed=H + 1, mask_frac=0.1)
    d, N, m, P = to_dev(p)
    d2, N2 = to_dev(q)[:2]
    args = (d, d2, N, N2, m, P, (0.2 * P).contiguous())
    many = wf.wf_sample_spin2(*args, seed=7, n_samples=2, n_chains=chains, burn_in=1, thin=2)
    for mode in ("auto", "global", "cluster"):
        prev = wf.wf_set_large_image_sampler(mode)
        try:
            one = wf.wf_sample_spin2(*args, seed=7, n_samples=2, chain_offset=chains - 1, burn_in=1, thin=2)
        finally:
            wf.wf_set_large_image_sampler(prev)
        assert rel(many[chains - 1].cpu().numpy(), one[0].cpu().numpy()) < 2e-6, (H, chains, mode)


def test_128_filter_starts_on_either_path():
    """A 128 x 128 filter from zero runs on the global-memory kernels, one with a starting iterate on chip: both reach
    the same map (to the refined tolerance, 1e-7 of the right-hand side in the residual norm)."""
    need_gpu()
    build.build()
    p = synth.config_paper128(3)
    dev = to_dev(p)
    r0 = wf.wf_solve_ex(*dev, tol=1e-7, refine=8)
    r1 = wf.wf_solve_ex(*dev, tol=1e-7, refine=8, init_s=(0.5 * dev[0]).contiguous())
    assert r0.resid < 1e-7 and r1.resid < 1e-7
    assert rel(r0.s.cpu().numpy(), r1.s.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("H,chains", [(128, 200), (64, 457), (32, 913)])
def test_shear_chains_in_balanced_shares(H, chains):
    """More pairs than are resident: the chains split between two CTAs equal the chains on their own (bit for bit:
    the same kernel, the state handed over in FP32)."""
    need_gpu()
    build.build()
    p, q = synth.make_problem(H, seed=H, mask_frac=0.1), synth.make_problem(H, seed=H + 1, mask_frac=0.1)
    d, N, m, P = to_dev(p)
    d2, N2 = to_dev(q)[:2]
    args = (d, d2, N, N2, m, P, (0.2 * P).contiguous())
    many = wf.wf_sample_spin2(*args, seed=7, n_samples=3, n_chains=chains, burn_in=1, thin=2)
    for c0 in range(0, chains, 152):   # these run one CTA per chain
        n = min(152, chains - c0)
        few = wf.wf_sample_spin2(*args, seed=7, n_samples=3, n_chains=n, chain_offset=c0, burn_in=1, thin=2)
        if H < 128 or n >= 40:
            assert torch.equal(many[c0:c0 + n], few)
        else:
            assert rel(many[c0:c0 + n].cpu().numpy(), few.cpu().numpy()) < 2e-6


@pytest.mark.parametrize("H,chains", [(128, 310), (128, 905), (32, 1600)])
def test_chains_and_bands_in_balanced_shares(H, chains):
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H, mask_frac=0.1)
    dev = to_dev(p)
    many = wf.wf_sample_ex(*dev, seed=7, n_samples=2, n_chains=chains, burn_in=2, thin=3)
    bins = (torch.arange(H * (H // 2 + 1), device="cuda", dtype=torch.int32) * 0).reshape(H, H // 2 + 1)
    ky = torch.fft.fftfreq(H, device="cuda").abs()[:, None] * H
    kx = torch.arange(H // 2 + 1, device="cuda")[None, :]
    bins += torch.sqrt(ky * ky + kx * kx).to(torch.int32).clamp(max=H // 2 - 1) - 1
    P0 = torch.ones(int(bins.max()) + 1, device="cuda")
    bs, bp = wf.wf_sample_band(*dev, bins.contiguous(), P0, seed=7, n_samples=2, n_chains=chains, burn_in=1, thin=2)
    for c0 in range(0, chains, 300):
        n = min(300, chains - c0)
        few = wf.wf_sample_ex(*dev, seed=7, n_samples=2, n_chains=n, chain_offset=c0, burn_in=2, thin=3)
        if H < 128 or n >= 36:
            assert torch.equal(many[c0:c0 + n], few)
        fs, fp = wf.wf_sample_band(*dev, bins.contiguous(), P0, seed=7, n_samples=2, n_chains=n, chain_offset=c0,
                                   burn_in=1, thin=2)
        assert torch.equal(bs[c0:c0 + n], fs) and torch.equal(bp[c0:c0 + n], fp)

"""Few large fields, a block of rows and columns per CTA for the whole launch (up to 256^2 in thread-block clusters),
against the same passes in the same order with several blocks per CTA: equal bit for bit, up to and past the number of
resident fields."""
import numpy as np
import pytest

from gpu_common import need_gpu, rel, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.fixture
def in_global():
    def f(call):
        wf.wf_set_large_image_sampler("global")
        try:
            return call()
        finally:
            wf.wf_set_large_image_sampler("auto")
    return f


@pytest.mark.parametrize("H,chains", [(128, 1), (128, 15), (128, 35), (128, 48), (128, 49), (256, 1), (256, 7),
                                      (256, 8), (256, 14), (256, 15), (512, 1), (512, 4), (512, 5), (1024, 1),
                                      (1024, 2)])
@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_samples_equal_global_memory(in_global, H, chains, dtype):
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H + chains, mask_frac=0.1)
    dev = to_dev(p)
    s0 = torch.randn(chains, H, H, device="cuda")
    out = torch.empty(chains, 2, H, H, device="cuda", dtype=getattr(torch, dtype))

    def call():
        wf.wf_sample_ex(*dev, seed=3, n_samples=2, n_chains=chains, chain_offset=5, start_step=7, burn_in=1, thin=2,
                        init_s=s0, out=out, out_dtype="f32" if dtype == "float32" else "bf16")
        return out.clone()

    a, b = call(), in_global(call)
    if H == 128 and chains > 47:  # the other side may be the on-chip kernel
        assert rel(a.float().cpu().numpy(), b.float().cpu().numpy()) < (2e-6 if dtype == "float32" else 2 ** -8)
    else:
        assert torch.equal(a, b)


@pytest.mark.parametrize("H", [128, 256, 512, 1024])
@pytest.mark.parametrize("check,refine", [(1, 0), (3, 0), (10, 2)])
def test_filter_equals_global_memory(in_global, H, check, refine):
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H, mask_frac=0.2, k0=1 / 32)
    dev = to_dev(p)
    call = lambda: wf.wf_solve_ex(*dev, tol=1e-5, check=check, refine=refine)
    a, b = call(), in_global(call)
    # the same states bit for bit; the residual adds the same terms in another order (FP32 within a thread)
    assert a.iters == b.iters
    assert abs(a.resid - b.resid) <= 1e-6 * b.resid
    if refine == 0:
        assert torch.equal(a.s, b.s)
    else:  # the FP64 residual's sums come from atomics
        assert rel(a.s.cpu().numpy(), b.s.cpu().numpy()) < 1e-6


@pytest.mark.parametrize("H,chains", [(128, 1), (128, 15), (128, 30), (256, 1), (256, 4), (256, 9), (256, 10), (512, 1), (512, 2),
                                      (512, 3)])
def test_shear_samples_equal_global_memory(in_global, H, chains):
    need_gpu()
    build.build()
    p, q = synth.make_problem(H, seed=H, mask_frac=0.1), synth.make_problem(H, seed=H + 1, mask_frac=0.1)
    d, N, m, P = to_dev(p)
    d2, N2 = to_dev(q)[:2]
    args = (d, d2, N, N2, m, P, (0.2 * P).contiguous())
    call = lambda: wf.wf_sample_spin2(*args, seed=3, n_samples=2, n_chains=chains, chain_offset=5, burn_in=1, thin=2)
    assert torch.equal(call(), in_global(call))


@pytest.mark.parametrize("H", [128, 256, 512])
def test_shear_filter_equals_global_memory(in_global, H):
    need_gpu()
    build.build()
    p, q = synth.make_problem(H, seed=H, mask_frac=0.1), synth.make_problem(H, seed=H + 1, mask_frac=0.1)
    d, N, m, P = to_dev(p)
    d2, N2 = to_dev(q)[:2]
    call = lambda: wf.wf_solve_spin2(d, d2, N, N2, m, P, (0.2 * P).contiguous(), tol=1e-5)
    a, b = call(), in_global(call)
    assert a.iters == b.iters and torch.equal(a.s, b.s)


@pytest.mark.parametrize("chains", [1, 7, 114, 115])
def test_64_in_clusters(chains):
    """64^2 in clusters of 4 CTAs (rows of 32 points: no middle pass) against the on-chip kernel: the same draws, FP32
    roundings apart; the sweeps contract, so the differences stay at a few units in the last place of the field."""
    need_gpu()
    build.build()
    p = synth.make_problem(64, seed=chains, mask_frac=0.1)
    dev = to_dev(p)
    s0 = torch.randn(chains, 64, 64, device="cuda")
    call = lambda: wf.wf_sample_ex(*dev, seed=3, n_samples=4, n_chains=chains, chain_offset=2, start_step=3, burn_in=1,
                                   thin=2, init_s=s0)
    a = call()
    wf.wf_set_large_image_sampler("global")  # on chip below 128
    try:
        b = call()
    finally:
        wf.wf_set_large_image_sampler("auto")
    assert rel(a.cpu().numpy(), b.cpu().numpy()) < 2e-6


@pytest.mark.parametrize("H,probes", [(32, 3), (32, 64), (32, 65), (64, 2), (64, 67), (128, 2), (128, 49), (256, 7),
                                      (256, 15), (512, 3)])
def test_probes_solved_side_by_side(in_global, H, probes):
    """The trace probes of the gradient, several solves in one launch (up to 64 on chip, else as many as are resident),
    against the batched gradient's own solves, and from 128 on against one solve after the other (the same iterates)."""
    need_gpu()
    build.build()
    p = synth.make_problem(H, seed=H, mask_frac=0.1, slope=-2.0, amp=1.2, k0=1.0 / H, sigma2=(0.01, 0.2))
    d, s2, m = to_dev(p)[:3]
    call = lambda: wf.wf_loglike_grad(d, s2, m, 1.2, -2.0, 1.0 / H, 1.0, n_probes=probes, seed=5, tol=1e-6)
    a = call()
    if H >= 128:
        b = in_global(call)
        np.testing.assert_allclose(a.grad, b.grad, rtol=1e-9)
        np.testing.assert_allclose(a.grad_var, b.grad_var, rtol=1e-6)
    c = wf.wf_loglike_grad_batch([(d, s2, m, 1.2, -2.0, 1.0 / H, 1.0, 5)], n_probes=probes, tol=1e-6)[0]
    # both solve to a relative residual of 1e-5
    sd = np.sqrt(a.grad_var) + 1e-12
    assert np.all(np.abs(c.grad - a.grad) < 0.05 * sd + 1e-3 * np.abs(a.grad))

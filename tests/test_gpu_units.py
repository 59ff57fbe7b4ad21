"""The refined Wiener filter and its derivatives do not depend on the unit of the data: with d in units of c, and the noise
variance and the spectrum in units of c^2, the map scales by c and the relative residual stays."""
import numpy as np
import pytest

from gpu_common import need_gpu, rel, to_dev, torch
from oracle import messenger as M
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu

UNITS = [1e-7, 1e-5, 1e6]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()
    build.build()


def _problem(H, c, amp=1.0):
    p = synth.make_problem(H, seed=H, mask_frac=0.1, k0=1.0 / 32, amp=amp)
    p.d = (p.d.astype(np.float64) * c).astype(np.float32)
    p.Ndiag = (p.Ndiag.astype(np.float64) * c * c).astype(np.float32)
    p.Pk = (p.Pk.astype(np.float64) * c * c).astype(np.float32)
    return p


@pytest.mark.parametrize("H", [16, 64, 128, 512])
@pytest.mark.parametrize("c,amp", [(c, 1.0) for c in UNITS] + [(1.0, 1e-6)])
def test_refined_filter_in_any_unit(H, c, amp):
    """The FP32 map's own rounding leaves a residual of a few 1e-8 (tol 1e-7 is reached in every unit), and bounds the
    difference of two units' maps: inputs and outputs are rounded once each in either unit (2^-24 = 6e-8 relative, times
    the few that the filter of a signal of this spectrum lets through)."""
    one = wf.wf_solve_ex(*to_dev(_problem(H, 1.0, amp)), tol=1e-7, refine=8)
    p = _problem(H, c, amp)
    r = wf.wf_solve_ex(*to_dev(p), tol=1e-7, refine=8, allow_not_converged=True)
    assert r.status == 0 and r.resid < 1e-7, (r.status, r.resid)
    s = r.s.double().cpu().numpy()
    rho = M.residual(s, p.d, p.Ndiag, p.mask, p.Pk)
    assert abs(rho - r.resid) <= 1e-3 * rho + 1e-13, (rho, r.resid)
    assert rel(s / c, one.s.double().cpu().numpy()) < 1e-6


@pytest.mark.parametrize("c", UNITS)
def test_wiener_map_in_any_unit(c):
    """The map of the differentiable form at its tolerance of 3e-8, with d, sigma2 and the amplitude in units of c, c^2, c^2."""
    H = 64
    p = synth.make_problem(H, seed=3, mask_frac=0.1, k0=1.0 / H, sigma2=(0.05, 0.3))

    def call(u):
        d = torch.from_numpy((p.d.astype(np.float64) * u).astype(np.float32)).cuda()
        s2 = torch.from_numpy((p.Ndiag.astype(np.float64) * u * u).astype(np.float32)).cuda()
        s, _ = wf.wf_wiener_vjp(d, s2, torch.from_numpy(p.mask).cuda(), 1.3 * u * u, -1.8, 1.0 / H, 0.9, tol=3e-8)
        return s.double().cpu().numpy() / u

    assert rel(call(c), call(1.0)) < 1e-6


@pytest.mark.parametrize("c", UNITS)
def test_vjp_in_any_unit(c):
    """d, sigma2 and the amplitude in units of c, c^2 and c^2: the map scales by c, its derivatives by c (slope, alpha) and
    1/c (amplitude). Solves to 3e-8, derivatives as sums over 64^2 modes and pixels of products of two such solutions."""
    H = 64
    p = synth.make_problem(H, seed=3, mask_frac=0.1, k0=1.0 / H, sigma2=(0.05, 0.3))
    g = torch.from_numpy(np.random.default_rng(H).standard_normal((H, H)).astype(np.float32)).cuda()

    def call(u):
        d = torch.from_numpy((p.d.astype(np.float64) * u).astype(np.float32)).cuda()
        s2 = torch.from_numpy((p.Ndiag.astype(np.float64) * u * u).astype(np.float32)).cuda()
        s, v = wf.wf_wiener_vjp(d, s2, torch.from_numpy(p.mask).cuda(), 1.3 * u * u, -1.8, 1.0 / H, 0.9, g, tol=3e-8)
        return s.double().cpu().numpy() / u, v * np.array([u, 1.0 / u, 1.0 / u])

    (s1, v1), (s, v) = call(1.0), call(c)
    assert rel(s, s1) < 1e-6
    np.testing.assert_allclose(v, v1, rtol=1e-4, atol=1e-6 * np.abs(v1).max())


@pytest.mark.parametrize("H", [16, 64, 256])
@pytest.mark.parametrize("c", UNITS)
def test_likelihood_gradient_in_any_unit(H, c):
    """Gradients by amplitude, slope and alpha scale by 1/c^2, 1 and 1. The trace probes' solves stop at 1e-5 in either
    unit (their sums agree to a few times that)."""
    p = synth.make_problem(H, seed=4, mask_frac=0.1, k0=1.0 / H, sigma2=(0.05, 0.3))

    def call(u, batch=False):
        d = torch.from_numpy((p.d.astype(np.float64) * u).astype(np.float32)).cuda()
        s2 = torch.from_numpy((p.Ndiag.astype(np.float64) * u * u).astype(np.float32)).cuda()
        m = torch.from_numpy(p.mask).cuda()
        par = (1.3 * u * u, -1.8, 1.0 / H, 0.9)
        if batch:
            r = wf.wf_loglike_grad_batch([(d, s2, m, *par, 1)], n_probes=3, tol=1e-6)[0]
        else:
            r = wf.wf_loglike_grad(d, s2, m, *par, n_probes=3, seed=1, tol=1e-6)
        return r.grad * np.array([u * u, 1.0, 1.0])

    one, got, batch = call(1.0), call(c), call(c, batch=True)
    np.testing.assert_allclose(got, one, rtol=1e-4, atol=1e-4 * np.abs(one).max())
    np.testing.assert_allclose(batch, one, rtol=1e-3, atol=1e-3 * np.abs(one).max())


@pytest.mark.parametrize("H,mode", [(16, "auto"), (64, "auto"), (128, "auto"), (128, "global"), (256, "auto"), (256, "global"),
                                    (256, "cluster"), (512, "auto"), (512, "cluster"), (1024, "auto")])
@pytest.mark.parametrize("c", [1e-12, 1e10])
def test_unrefined_filter_in_any_unit(H, mode, c):
    """The FP32 iteration stops by the level norms ||S N^-1 d||^2, which have the unit of the map squared. Two maps that stop
    at a residual of 1e-5 differ by a few times that."""
    wf.wf_set_large_image_sampler(mode)
    try:
        one = wf.wf_solve_ex(*to_dev(_problem(H, 1.0)), tol=1e-5, refine=0)
        r = wf.wf_solve_ex(*to_dev(_problem(H, c)), tol=1e-5, refine=0)
    finally:
        wf.wf_set_large_image_sampler("auto")
    assert abs(r.iters - one.iters) <= 4, (r.iters, one.iters)
    assert rel(r.s.double().cpu().numpy() / c, one.s.double().cpu().numpy()) < 1e-4


@pytest.mark.parametrize("small_path", [0, 1])
@pytest.mark.parametrize("c", [1e-12, 1e10])
def test_batch_in_any_unit(small_path, c):
    sizes = [16, 32, 64, 128, 256, 512]

    def call(u):
        images = [wf.BatchImage(*to_dev(_problem(H, u))) for H in sizes]
        wf.wf_batch_run(images, small_path=small_path)
        return images

    for a, b in zip(call(c), call(1.0)):
        assert abs(a.iters - b.iters) <= 4, (a.iters, b.iters)
        assert rel(a.out_wf.double().cpu().numpy() / c, b.out_wf.double().cpu().numpy()) < 1e-4

"""GPU checks of the FP64 transforms behind the residuals and the mass mapping, at the sizes and field counts where
they change shape (rows per CTA, radix-2 pass, several chunks of fields)."""
import numpy as np
import pytest

from gpu_common import need_gpu, rel, to_dev, torch
from oracle import messenger as M, spin2 as S2
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()
    build.build()


@pytest.mark.parametrize("H", [16, 32, 64, 128, 512, 1024])
def test_convergence_sizes(H):
    """The FP32 outputs are rounded once from FP64, so 1e-7 relative L2 bounds them (half an ulp, 6e-8)."""
    g = np.random.default_rng(H).standard_normal((3, 2, H, H)).astype(np.float32)
    k = wf.wf_shear_to_convergence(torch.from_numpy(g).cuda()).cpu().numpy()
    for i in range(3):
        kE, kB = S2.convergence_from_shear(g[i, 0], g[i, 1])
        assert rel(k[i, 0], kE) < 1e-7 and rel(k[i, 1], kB) < 1e-7


def test_convergence_of_more_fields_than_one_chunk():
    """16384 fields of 16 x 16 fill a chunk: the fields of a longer call equal those of calls of their own."""
    g = torch.randn((16384 + 3, 2, 16, 16), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    k = wf.wf_shear_to_convergence(g)
    for sl in (slice(0, 5), slice(16380, 16387)):
        assert torch.equal(k[sl], wf.wf_shear_to_convergence(g[sl].contiguous()))


@pytest.mark.parametrize("H", [16, 128, 512])
def test_refined_filter_with_response_and_empty_modes(H):
    """Corrections at tol 1e-8 with a pixel response and modes without power: the reported residual is the oracle's
    residual of the returned map (to 1e-3 of itself, plus FP64 rounding)."""
    p = synth.make_problem(H, seed=H, mask_frac=0.1, slope=-1.0, k0=1.0 / 8)
    p.Pk[:, H // 4] = 0.0
    rng = np.random.default_rng(H + 1)
    A = rng.uniform(0.5, 1.5, (H, H)).astype(np.float32)
    A[1, 2] = 0.0
    r = wf.wf_solve_ex(*to_dev(p), tol=1e-8, refine=8, A=torch.from_numpy(A).cuda(), allow_not_converged=True)
    rho = M.residual(r.s.double().cpu().numpy(), p.d, p.Ndiag, p.mask, p.Pk, A=A)
    assert abs(rho - r.resid) <= 1e-3 * rho + 1e-13, (rho, r.resid)
    assert r.resid < 1e-7

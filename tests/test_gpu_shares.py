"""Equal shares only where they are faster than one CTA per chain."""
import ctypes
import time

import pytest

from gpu_common import need_gpu, to_dev, torch
from paper_1810_02821_gb300 import build, synth, wf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains", [3000, 5000])
def test_full_rounds_are_not_shared_out(chains):
    """32 x 32, last rounds of 0.97 and 0.29 of the resident chains: the sampler takes no longer than the form without
    device allocation, which always runs one CTA per chain (shares took 6% longer). Time per sweep from calls of 100 and 500
    sweeps, the median of nine each, in turn."""
    need_gpu()
    build.build()
    dev = to_dev(synth.make_problem(32, seed=3, mask_frac=0.1, k0=1.0 / 32))
    out = torch.empty(chains, 1, 32, 32, device="cuda")
    lib = wf.load_library()
    plain_call = lib.wf_sample_noalloc
    plain_call.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int32, ctypes.c_int32, ctypes.c_uint64,
                                                  ctypes.POINTER(wf.SampleOpts), ctypes.c_void_p, ctypes.c_void_p]
    plain_call.restype = ctypes.c_int
    o = wf.SampleOpts()
    lib.wf_sample_opts_default(ctypes.byref(o))
    o.n_samples, o.n_chains = 1, chains

    def without_allocation(thin):
        o.thin = thin
        assert plain_call(*[x.data_ptr() for x in dev], 32, 32, 5, ctypes.byref(o), out.data_ptr(),
                          torch.cuda.current_stream().cuda_stream) == 0

    calls = [lambda thin: wf.wf_sample_ex(*dev, seed=5, n_samples=1, n_chains=chains, thin=thin, out=out), without_allocation]
    t = {}
    for i in range(10):
        for k, call in enumerate(calls):
            for thin in (100, 500):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                call(thin)
                torch.cuda.synchronize()
                t.setdefault((k, thin), []).append(time.perf_counter() - t0)
    med = {key: sorted(x[1:])[4] for key, x in t.items()}
    ex, plain = (1e6 * (med[k, 500] - med[k, 100]) / 400 for k in (0, 1))
    print(f"{chains} chains: {ex:.2f} us a sweep, one CTA per chain {plain:.2f} us")
    assert ex < 1.04 * plain


@pytest.mark.parametrize("kind,H,chains,sweeps", [("sample", 128, 310, 14), ("sample", 128, 615, 14), ("sample", 32, 1600, 60),
                                                  ("band", 128, 310, 30), ("band", 64, 770, 30), ("band", 32, 1600, 30),
                                                  ("shear", 128, 200, 14), ("shear", 64, 457, 20), ("shear", 32, 913, 60)])
def test_calls_long_enough_to_share_out(kind, H, chains, sweeps):
    """Chains split between two CTAs equal the same chains in calls of one round (the same kernel, the state handed over in
    FP32: bit for bit); from 36 (shear 40) chains a call, below which few 128 x 128 fields run another kernel."""
    need_gpu()
    build.build()
    p, q = synth.make_problem(H, seed=H, mask_frac=0.1), synth.make_problem(H, seed=H + 1, mask_frac=0.1)
    d, N, m, P = to_dev(p)
    d2, N2 = to_dev(q)[:2]
    ky = torch.fft.fftfreq(H, device="cuda").abs()[:, None] * H
    kx = torch.arange(H // 2 + 1, device="cuda")[None, :]
    bins = (torch.sqrt(ky * ky + kx * kx).to(torch.int32).clamp(max=H // 2 - 1) - 1).contiguous()
    P0 = torch.ones(int(bins.max()) + 1, device="cuda")
    o = dict(n_samples=2, burn_in=sweeps % 2, thin=sweeps // 2)

    def call(n, c0):
        if kind == "sample":
            return (wf.wf_sample_ex(d, N, m, P, seed=7, n_chains=n, chain_offset=c0, **o),)
        if kind == "band":
            return wf.wf_sample_band(d, N, m, P, bins, P0, seed=7, n_chains=n, chain_offset=c0, **o)
        return (wf.wf_sample_spin2(d, d2, N, N2, m, P, (0.2 * P).contiguous(), seed=7, n_chains=n, chain_offset=c0, **o),)

    many = call(chains, 0)
    step = chains // 8 + 1 if chains // 8 >= 52 else 60
    for c0 in range(0, chains - step + 1, step):
        for a, b in zip(many, call(step, c0)):
            assert torch.equal(a[c0:c0 + step], b)
    for a, b in zip(many, call(step, chains - step)):
        assert torch.equal(a[chains - step:], b)

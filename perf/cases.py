"""Performance cases of the messenger-field Wiener filter and samplers.

Each case is one call (or one pair of calls that a program makes together) through the public binding
``paper_1810_02821_gb300.wf``, on inputs of the data model d = A s + n: a Gaussian random field with a
power-law spectrum, spatially varying noise variance, a mask of missing pixels and, where stated, a
diagonal pixel response A. Inputs are made on the GPU from the seed alone.

``exact`` restates each computation in plain torch in FP64: the Philox4x32-10 counter layout of the draws,
Alg. 1 with an FFT, and conjugate gradients for the Wiener filter.
"""
from __future__ import annotations

import math

import torch

DEV = "cuda"
F64 = torch.float64


# ----------------------------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a few posterior draws of a 32 x 32 image, as in an interactive program or an
        # inner loop of a larger inference; latency and launches count
        dict(name="sample_32_one", kind="sample", size=32, chains=1, samples=16, thin=1, burn_in=0, out="f32", response=False),
        # the paper's own use: one long chain of a 128 x 128 image, thinned
        dict(name="sample_128_one", kind="sample", size=128, chains=1, samples=50, thin=4, burn_in=0, out="f32", response=False),
        # many chains of one 128 x 128 image (production sampling; a count that is no multiple of the GPU)
        dict(name="sample_128_many", kind="sample", size=128, chains=1000, samples=10, thin=4, burn_in=0, out="f32", response=False),
        # a few chains of a larger survey patch, after burn-in
        dict(name="sample_256_few", kind="sample", size=256, chains=3, samples=20, thin=2, burn_in=10, out="f32", response=False),
        # many chains of a 512 x 512 image with the samples kept as BF16 (storage-bound analyses)
        dict(name="sample_512_many", kind="sample", size=512, chains=50, samples=8, thin=2, burn_in=0, out="bf16", response=False),
        # a small Wiener filter with a pixel response: one call per small image
        dict(name="solve_64", kind="solve", size=64, tol=1e-6, precision=False, response=True),
        # a large Wiener filter on the precision problem (noise variance over two decades, holes over 20% of
        # the area)
        dict(name="solve_1024", kind="solve", size=1024, tol=1e-6, precision=True, response=False),
        # power-spectrum inference: the hierarchical sampler with radial bands
        dict(name="band_128", kind="band", size=128, chains=300, samples=15, thin=2, bands=90),
        # mass mapping by sampling: shear draws for a set of chains
        dict(name="shear_128", kind="shear", size=128, chains=200, samples=15, thin=2),
        # mass mapping by filtering: the shear Wiener filter, then the convergence maps of the filtered shear
        dict(name="mass_map_256", kind="mass_map", size=256, tol=1e-5),
        # a catalogue of cut-outs of mixed sizes, filtered and sampled in one call
        dict(name="batch_mixed", kind="batch", images=512, samples=16),
        # gradient-based inference of the spectrum and noise parameters: log-likelihood gradient (forward
        # solve and trace probes), then the vector-Jacobian product of the Wiener map (adjoint solve)
        dict(name="gradient_256", kind="gradient", size=256, probes=4, tol=1e-6),
    ]


def draw(rng):
    kind = rng.choice(["sample", "sample", "sample", "solve", "solve", "band", "shear", "mass_map", "batch", "gradient"])

    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))

    if kind == "sample":
        size = rng.choice([16, 32, 64, 128, 128, 256, 512, 1024])
        thin, burn_in = rng.choice([1, 1, 2, 3, 5]), rng.choice([0, 0, 3, 10])
        samples = log_int(1, 40)
        sweeps = burn_in + thin * samples
        budget = 6.0e8 if size <= 256 else 2.0e8  # pixels times sweeps: within the listed cases
        most = max(1, min(2000, int(budget / (size * size * sweeps))))
        return dict(kind=kind, size=size, chains=log_int(1, most), samples=samples, thin=thin, burn_in=burn_in,
                    out=rng.choice(["f32", "f32", "bf16", "f16"]), response=rng.random() < 0.25)
    if kind == "solve":
        size = rng.choice([16, 32, 64, 128, 256, 512, 1024])
        return dict(kind=kind, size=size, tol=rng.choice([1e-5, 1e-6]), precision=rng.random() < 0.4,
                    response=rng.random() < 0.3)
    if kind == "band":
        size = rng.choice([32, 64, 128, 256, 512])
        samples, thin = log_int(1, 20), rng.choice([1, 2, 3])
        most = max(1, min(600, int(1.4e8 / (size * size * samples * thin))))
        return dict(kind=kind, size=size, chains=log_int(1, most), samples=samples, thin=thin,
                    bands=rng.randint(3, min(256, 7 * size // 10)))
    if kind == "shear":
        size = rng.choice([32, 64, 128, 256, 512])
        samples, thin = log_int(1, 20), rng.choice([1, 2, 3])
        most = max(1, min(400, int(1.0e8 / (size * size * samples * thin))))
        return dict(kind=kind, size=size, chains=log_int(1, most), samples=samples, thin=thin)
    if kind == "mass_map":
        return dict(kind=kind, size=rng.choice([32, 64, 128, 256]), tol=rng.choice([1e-4, 1e-5]))
    if kind == "batch":
        return dict(kind=kind, images=log_int(5, 500), samples=rng.randint(1, 16))
    return dict(kind=kind, size=rng.choice([32, 64, 128, 256]), probes=rng.randint(1, 4), tol=1e-6)


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=F64)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=F64)


def _uniform(g, lo, hi):
    return lo + (hi - lo) * float(_rand(g, 1)[0])


def _wavenumber(n):
    ky = torch.fft.fftfreq(n, device=DEV, dtype=F64)[:, None]
    kx = (torch.arange(n // 2 + 1, device=DEV, dtype=F64) / n)[None, :]
    return torch.sqrt(ky * ky + kx * kx)


def _power_law(n, amp, slope, k0):
    """P(k) = amp (k / k0)^slope on the half spectrum, 0 at k = 0 (variance of the unitary transform)."""
    k = _wavenumber(n)
    k[0, 0] = 1.0
    p = amp * (k / k0) ** slope
    p[0, 0] = 0.0
    return p.float()


def _field(P, n, g):
    w = torch.fft.rfft2(_randn(g, n, n), norm="ortho") * torch.sqrt(P.double())
    return torch.fft.irfft2(w, s=(n, n), norm="ortho")


def _scatter_mask(n, frac, g):
    return (_rand(g, n, n) < frac).to(torch.uint8)


def _hole_mask(n, g):
    """Circular holes (periodic) with radii n/256 .. 3n/100 covering about a fifth of the area."""
    mask = torch.zeros(n, n, dtype=torch.bool, device=DEV)
    c = (_rand(g, 200, 2) * n).cpu()
    r = (n / 256 + (0.03 * n - n / 256) * _rand(g, 200)).cpu()
    x = torch.arange(n, device=DEV, dtype=F64) + 0.5
    for i in range(200):
        dy = (x - float(c[i, 0])).abs()
        dx = (x - float(c[i, 1])).abs()
        dy, dx = torch.minimum(dy, n - dy), torch.minimum(dx, n - dx)
        mask |= dy[:, None] ** 2 + dx[None, :] ** 2 <= float(r[i]) ** 2
    return mask.to(torch.uint8)


def _image(n, seed, salt=0, slope=-2.0, amp=1.0, k0=1.0 / 32, sigma2=(0.05, 0.5), mask_frac=0.1, holes=False,
           response=False):
    g = _gen(seed, salt)
    P = _power_law(n, amp, slope, k0)
    s = _field(P, n, g)
    N = sigma2[0] + (sigma2[1] - sigma2[0]) * _rand(g, n, n)
    mask = _hole_mask(n, g) if holes else _scatter_mask(n, mask_frac, g)
    A = None
    if response:  # gains around one, a few dead pixels
        A = (0.4 + 1.2 * _rand(g, n, n)) * (_rand(g, n, n) > 0.005)
        A = A.float()
        s = s * A.double()
    d = s + _randn(g, n, n) * torch.sqrt(N)
    d = torch.where(mask != 0, torch.zeros_like(d), d)
    return dict(d=d.float(), N=N.float(), mask=mask, P=P, A=A)


def _radial_bins(n, bands):
    """`bands` bins of equal width in radius up to the Nyquist radius, modes beyond it in the last; k = 0 out."""
    ky = torch.fft.fftfreq(n, device=DEV, dtype=F64)[:, None] * n
    kx = torch.arange(n // 2 + 1, device=DEV, dtype=F64)[None, :]
    r = torch.sqrt(ky * ky + kx * kx)
    b = torch.clamp(torch.floor((r - 1.0) * bands / (n / math.sqrt(2.0))), 0, bands - 1).to(torch.int32)
    b[0, 0] = -1
    return b.contiguous()


SIZES = ((64, 0.40), (128, 0.40), (256, 0.15), (512, 0.05))


def _batch_images(case, seed):
    """Images per size (largest-remainder rounding of the fractions), each with its own spectrum, noise
    range and mask, in a random order."""
    m = case["images"]
    raw = [(n, m * f) for n, f in SIZES]
    count = {n: int(math.floor(x)) for n, x in raw}
    for n, _ in sorted(raw, key=lambda t: -(t[1] - math.floor(t[1])))[: m - sum(count.values())]:
        count[n] += 1
    g = _gen(seed, 99)
    groups = []
    for n, _ in SIZES:
        c = count[n]
        if c == 0:
            continue
        u = _rand(g, 4, c)
        slope = -3.0 + 2.0 * u[0]
        lo = 0.01 + 0.09 * u[1]
        hi = lo * (2.0 + 18.0 * u[2])
        k = _wavenumber(n)
        k[0, 0] = 1.0
        P = (k[None] * n) ** slope[:, None, None]
        P[:, 0, 0] = 0.0
        P = P.float().contiguous()
        s = torch.fft.irfft2(torch.fft.rfft2(_randn(g, c, n, n), norm="ortho") * torch.sqrt(P.double()), s=(n, n),
                             norm="ortho")
        N = lo[:, None, None] + (hi - lo)[:, None, None] * _rand(g, c, n, n)
        mask = _rand(g, c, n, n) < (0.1 * u[3])[:, None, None]
        h = max(1, n // 6)  # and one rectangle
        at = (_rand(g, c, 2) * n).long()
        x = torch.arange(n, device=DEV)
        iny = ((x[None, :] - at[:, :1]) % n) < h
        inx = ((x[None, :] - at[:, 1:]) % n) < h
        mask |= iny[:, :, None] & inx[:, None, :]
        d = torch.where(mask, torch.zeros_like(s), s + _randn(g, c, n, n) * torch.sqrt(N))
        groups.append(dict(size=n, count=c, d=d.float(), N=N.float(), mask=mask.to(torch.uint8), P=P))
    order = torch.randperm(sum(q["count"] for q in groups), generator=_gen(seed, 98), device=DEV).cpu().tolist()
    return groups, order


def _inputs(case, seed):
    kind = case["kind"]
    if kind == "sample":
        return _image(case["size"], seed, response=case["response"])
    if kind == "solve":
        if case["precision"]:
            return _image(case["size"], seed, slope=-1.5, sigma2=(0.001, 0.1), holes=True, response=case["response"])
        return _image(case["size"], seed, response=case["response"])
    if kind == "band":
        q = _image(case["size"], seed, sigma2=(0.01, 1.0))
        q["bins"] = _radial_bins(case["size"], case["bands"])
        q["P0"] = torch.ones(case["bands"], device=DEV)
        return q
    if kind in ("shear", "mass_map"):
        n = case["size"]
        g = _gen(seed, 7)
        PE = _power_law(n, 1.0, -2.0, 1.0 / 32)
        PB = (0.2 * PE).float().contiguous()
        c, s = _rotation(n)
        e = torch.fft.rfft2(_field(PE, n, g), norm="ortho")
        b = torch.fft.rfft2(_field(PB, n, g), norm="ortho")
        g1 = torch.fft.irfft2(c * e - s * b, s=(n, n), norm="ortho")
        g2 = torch.fft.irfft2(s * e + c * b, s=(n, n), norm="ortho")
        mask = _scatter_mask(n, 0.1, g)
        N1, N2 = (0.05 + 0.45 * _rand(g, n, n)), (0.05 + 0.45 * _rand(g, n, n))
        z = torch.zeros_like(g1)
        d1 = torch.where(mask != 0, z, g1 + _randn(g, n, n) * torch.sqrt(N1))
        d2 = torch.where(mask != 0, z, g2 + _randn(g, n, n) * torch.sqrt(N2))
        return dict(d1=d1.float(), d2=d2.float(), N1=N1.float(), N2=N2.float(), mask=mask, PE=PE, PB=PB)
    if kind == "gradient":
        g = _gen(seed, 5)
        amp, slope = _uniform(g, 0.5, 2.0), _uniform(g, -2.5, -1.5)
        q = _image(case["size"], seed, salt=6, slope=slope, amp=amp, k0=1.0 / case["size"], sigma2=(0.01, 0.2))
        q.update(amp=amp, slope=slope, k0=1.0 / case["size"], alpha=1.0,
                 g=_randn(g, case["size"], case["size"]).float())
        return q
    raise ValueError(kind)


# ----------------------------------------------------------------------------------------------
# the framework
# ----------------------------------------------------------------------------------------------
OUT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def prepare(case, seed):
    from paper_1810_02821_gb300 import wf
    kind = case["kind"]
    if kind == "batch":
        groups, order = _batch_images(case, seed)
        images = []
        for q in groups:
            n, c, m = q["size"], q["count"], case["samples"]
            q["wf"] = torch.empty(c, n, n, device=DEV)
            q["s"] = torch.empty(c, m, n, n, device=DEV)
            for i in range(c):
                images.append(wf.BatchImage(q["d"][i], q["N"][i], q["mask"][i], q["P"][i], seed=seed, chain=len(images),
                                            out_wf=q["wf"][i], out_samples=q["s"][i]))
        return dict(case=case, groups=groups, images=[images[i] for i in order])
    st = _inputs(case, seed)
    st.update(case=case, seed=int(seed) + 12345)
    n = case.get("size")
    if kind == "sample":  # a program keeps the buffer that its samples land in
        st["out"] = torch.empty(case["chains"], case["samples"], n, n, dtype=OUT[case["out"]], device=DEV)
    return st


def run(state):
    from paper_1810_02821_gb300 import wf
    c = state["case"]
    kind = c["kind"]
    if kind == "sample":
        return wf.wf_sample_ex(state["d"], state["N"], state["mask"], state["P"], state["seed"], c["samples"],
                               n_chains=c["chains"], burn_in=c["burn_in"], thin=c["thin"], A=state["A"],
                               out_dtype=c["out"], out=state["out"])
    if kind == "solve":
        return wf.wf_solve_ex(state["d"], state["N"], state["mask"], state["P"], tol=c["tol"], A=state["A"]).s
    if kind == "band":
        return wf.wf_sample_band(state["d"], state["N"], state["mask"], state["P"], state["bins"], state["P0"],
                                 state["seed"], c["samples"], n_chains=c["chains"], thin=c["thin"])
    if kind == "shear":
        return wf.wf_sample_spin2(state["d1"], state["d2"], state["N1"], state["N2"], state["mask"], state["PE"],
                                  state["PB"], state["seed"], c["samples"], n_chains=c["chains"], thin=c["thin"])
    if kind == "mass_map":
        s = wf.wf_solve_spin2(state["d1"], state["d2"], state["N1"], state["N2"], state["mask"], state["PE"],
                              state["PB"], tol=c["tol"]).s
        return s, wf.wf_shear_to_convergence(s)
    if kind == "batch":
        wf.wf_batch_run(state["images"], n_samples=c["samples"])
        return [(q["wf"], q["s"]) for q in state["groups"]]
    if kind == "gradient":
        par = (state["amp"], state["slope"], state["k0"], state["alpha"])
        r = wf.wf_loglike_grad(state["d"], state["N"], state["mask"], *par, n_probes=c["probes"], seed=state["seed"],
                               tol=c["tol"])
        s, v = wf.wf_wiener_vjp(state["d"], state["N"], state["mask"], *par, state["g"], s_w=r.wf, tol=c["tol"])
        return r.quad, r.grad_quad, r.grad, s, v
    raise ValueError(kind)


def work(case):
    """Bytes: each input once, each output once. Flops: the two real 2D transforms of a sweep, 5 n log2 n, and
    the draws at about 10 operations a variate (two variates a pixel and sweep); a Wiener filter counts the
    sweeps of the cooling schedule at its least (the levels from max P / tau to 1, one check each)."""
    kind = case["kind"]

    def sweeps(n, count, normals=2):
        return count * (5.0 * n * math.log2(n) + 10.0 * normals * n)

    def levels(pmax, tau):
        return 1 + max(0, math.ceil(math.log2(max(1.0, pmax / tau))))

    if kind == "batch":
        b = f = 0.0
        for h, frac in SIZES:
            n, m = h * h, case["images"] * frac
            b += m * n * (4 + 4 + 1 + 2 + 4 + 4 * case["samples"])
            f += m * (sweeps(n, case["samples"]) + sweeps(n, 4 * levels(1.0, 0.05), 0))
        return dict(bytes=b, flops=f)
    h = case["size"]
    n = h * h
    inp = n * (4 + 4 + 1 + 2) + 2 * h
    pmax = (32.0 / h) ** -2.0
    if kind == "sample":
        count = case["chains"] * (case["burn_in"] + case["samples"] * case["thin"])
        eb = 4 if case["out"] == "f32" else 2
        return dict(bytes=inp + eb * n * case["chains"] * case["samples"], flops=sweeps(n, count))
    if kind == "solve":
        lv = levels((32.0 / h) ** -1.5, 0.001) if case["precision"] else levels(pmax, 0.05)
        return dict(bytes=inp + 4 * n, flops=sweeps(n, 4 * lv, 0))
    if kind == "band":
        count = case["chains"] * case["samples"] * case["thin"]
        return dict(bytes=inp + 4 * n * case["chains"] * case["samples"], flops=sweeps(n, count, 3))
    if kind == "shear":
        count = 2 * case["chains"] * case["samples"] * case["thin"]
        return dict(bytes=2 * inp + 8 * n * case["chains"] * case["samples"], flops=sweeps(n, count))
    if kind == "mass_map":
        return dict(bytes=2 * inp + 16 * n, flops=2 * sweeps(n, 16 * levels(pmax, 0.05), 0))
    solves = 2 + case["probes"]
    return dict(bytes=inp + 12 * n, flops=sweeps(n, solves * 4 * levels(1.0, 0.01), 0))


def tolerance(case):
    kind = case["kind"]
    if kind in ("sample", "shear"):
        if case.get("out", "f32") != "f32":  # a stored value lands on the other side of a rounding now and then
            return dict(rel=3e-4, max=2e-2)
        return dict(rel=2e-6, max=2e-4)  # seen against exact(): 4e-7
    if kind == "band":  # the power of a band with few modes is a quotient by a small chi-square (seen: 4e-4)
        return dict(rel=1.5e-3, max=6e-2)
    if kind == "batch":  # the filter stops on its own FP32 residual, 1e-5 (seen: 1.6e-5)
        return dict(rel=1e-4, max=1e-2)
    if kind == "gradient":  # the trace probes' solves stop at 1e-5 (seen: 7e-5)
        return dict(rel=4e-4, max=1e-2)
    if kind == "solve" and case["precision"]:  # error of the map at residual tol, condition about 1e5
        return dict(rel=100 * case["tol"], max=1e-2)
    return dict(rel=10 * case["tol"], max=1e-2)


# ----------------------------------------------------------------------------------------------
# FP64 restatement
# ----------------------------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _mulhilo(a, x):
    lo = (a * x) & M32
    hi = (a * (x >> 16) + ((a * (x & 0xFFFF)) >> 16)) >> 16
    return hi, lo


def _philox(c0, c1, c2, c3, key):
    k0, k1 = key & M32, (key >> 32) & M32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c0)
        h1, l1 = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _words(groups, step, chains, stream, key):
    g = torch.arange(groups, device=DEV, dtype=torch.int64)[None, :].expand(len(chains), groups)
    ch = torch.as_tensor(chains, device=DEV, dtype=torch.int64)[:, None].expand(len(chains), groups)
    return _philox(g, torch.full_like(g, step), ch, torch.full_like(g, stream), key)


def _normals(groups, step, chains, stream, key):
    w = _words(groups, step, chains, stream, key)
    u = [(2.0 * (x >> 9).double() + 1.0) * 2.0 ** -24 for x in w]
    z = []
    for a, b in ((0, 1), (2, 3)):
        r = torch.sqrt(-2.0 * torch.log(u[a]))
        z += [r * torch.cos(2 * math.pi * u[b]), r * torch.sin(2 * math.pi * u[b])]
    return torch.stack(z, dim=-1)  # [chains][groups][4]


def _xi(n, step, chains, stream, key):
    return _normals(n * n // 4, step, chains, stream, key).reshape(len(chains), n, n)


def _zeta(n, step, chains, stream, key):
    """Hermitian white noise on the half spectrum [chains][n][n/2+1] in the counter layout of the s-draw."""
    h = n // 2
    z = _normals(h * h, step, chains, stream, key).reshape(len(chains), h, h, 4)  # [column][group j]
    a = torch.complex(z[..., 0], z[..., 1]) / math.sqrt(2.0)
    b = torch.complex(z[..., 2], z[..., 3]) / math.sqrt(2.0)
    out = torch.zeros(len(chains), n, h + 1, dtype=torch.complex128, device=DEV)
    out[:, :h, 1:h] = a[:, 1:, :].transpose(1, 2)
    out[:, h, 1:h] = b[:, 1:, 0]
    out[:, h + 1:, 1:h] = b[:, 1:, 1:].flip(2).transpose(1, 2)
    for col, v in ((0, a), (h, b)):
        out[:, 1:h, col] = v[:, 0, 1:]
        out[:, h + 1:, col] = v[:, 0, 1:].conj().flip(1)
    for i, (y, x) in enumerate(((0, 0), (h, 0), (0, h), (h, h))):
        out[:, y, x] = z[:, 0, 0, i].to(torch.complex128)
    return out


def _data(q):
    """(data, noise variance, observed) in FP64 of the A = I problem that a response reduces to."""
    d, N, obs = q["d"].double(), q["N"].double(), q["mask"] == 0
    if q.get("A") is not None:
        A = q["A"].double()
        obs = obs & (A != 0)
        A = torch.where(obs, A, torch.ones_like(A))
        d, N = d / A, N / (A * A)
    return d, N, obs


def _t_terms(d, N, obs, tau):
    """mean = a + w s and standard deviation of the t-draw."""
    w = torch.where(obs, (N - tau) / N, torch.ones_like(N)).clamp(min=0.0)
    a = torch.where(obs, (1.0 - w) * d, torch.zeros_like(d))
    return a, w, torch.sqrt(tau * w)


def _rfft(x):
    return torch.fft.rfft2(x, norm="ortho")


def _irfft(x, n):
    return torch.fft.irfft2(x, s=(n, n), norm="ortho")


def _rotation(n):
    ky = torch.fft.fftfreq(n, device=DEV, dtype=F64)[:, None] * n
    kx = torch.arange(n // 2 + 1, device=DEV, dtype=F64)[None, :]
    kk = kx * kx + ky * ky
    kk[0, 0] = 1.0
    c, s = (kx * kx - ky * ky) / kk, 2.0 * kx * ky / kk
    c[0, 0], s[0, 0] = 1.0, 0.0
    c[n // 2], s[n // 2] = 1.0, 0.0
    c[:, n // 2], s[:, n // 2] = 1.0, 0.0
    return c, s


def _cg(apply_S, d, N, obs, rel=1e-13, most=20000):
    """s = S C^-1 d over the observed pixels, C = S + N, by conjugate gradients on
    I + N^-1/2 S N^-1/2, for a batch of systems (sums over all dims but the first); and x = C^-1 d."""
    dims = tuple(range(1, d.dim()))
    si = torch.where(obs, 1.0 / torch.sqrt(torch.where(obs, N, torch.ones_like(N))), torch.zeros_like(N))

    def dot(a, b):
        return (a * b).sum(dims, keepdim=True)

    b = si * d
    u = torch.zeros_like(b)
    r, p = b.clone(), b.clone()
    rr = dot(r, r)
    stop = rel * rel * rr.clamp(min=1e-300)
    for i in range(most):
        Ap = p + si * apply_S(si * p)
        alpha = rr / dot(p, Ap).clamp(min=1e-300)
        u, r = u + alpha * p, r - alpha * Ap
        new = dot(r, r)
        p = r + (new / rr.clamp(min=1e-300)) * p
        rr = new
        if i % 20 == 19 and bool((rr <= stop).all()):
            break
    x = si * u
    return apply_S(x), x


def _scalar_S(P, n):
    P = P.double()
    return lambda v: _irfft(P * _rfft(v), n)


def _chain(s, q_terms, P, tau, n, steps, chains, key, keep):
    """Alg. 1 sweeps from s [chains][n][n]; keep(i, s) after each."""
    a, w, sd = q_terms
    f, gs = P / (P + tau), torch.sqrt(P * tau / (P + tau))
    for i in range(steps):
        t = a + w * s + sd * _xi(n, i, chains, 0, key)
        s = _irfft(f * _rfft(t) + gs * _zeta(n, i, chains, 1, key), n)
        keep(i + 1, s)
    return s


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    n = case["size"]
    q = _inputs(case, seed)
    key = int(seed) + 12345
    if kind == "sample":
        d, N, obs = _data(q)
        tau, P = float(N[obs].min()), q["P"].double()
        chains = list(range(case["chains"]))
        out = torch.empty(len(chains), case["samples"], n, n, dtype=F64, device=DEV)

        def keep(i, s):
            if i > case["burn_in"] and (i - case["burn_in"]) % case["thin"] == 0:
                out[:, (i - case["burn_in"]) // case["thin"] - 1] = s

        _chain(torch.zeros(len(chains), n, n, dtype=F64, device=DEV), _t_terms(d, N, obs, tau), P, tau, n,
               case["burn_in"] + case["samples"] * case["thin"], chains, key, keep)
        return out
    if kind == "solve":
        d, N, obs = _data(q)
        return _cg(_scalar_S(q["P"], n), d[None], N[None], obs[None])[0][0]
    if kind == "band":
        return _exact_band(case, q, key)
    if kind == "shear":
        return _exact_shear(case, q, key)
    if kind == "mass_map":
        c, s = _rotation(n)
        PE, PB = q["PE"].double(), q["PB"].double()

        def S(v):  # [1][2][n][n]
            a, b = _rfft(v[:, 0]), _rfft(v[:, 1])
            e, m = PE * (c * a + s * b), PB * (c * b - s * a)
            return torch.stack((_irfft(c * e - s * m, n), _irfft(s * e + c * m, n)), 1)

        d = torch.stack((q["d1"], q["d2"]))[None].double()
        N = torch.stack((q["N1"], q["N2"]))[None].double()
        obs = (q["mask"] == 0)[None, None].expand_as(d)
        g = _cg(S, d, N, obs)[0][0]
        a, b = _rfft(g[0]), _rfft(g[1])
        return g, torch.stack((_irfft(c * a + s * b, n), _irfft(c * b - s * a, n)))
    if kind == "gradient":
        return _exact_gradient(case, q, key)
    raise ValueError(kind)


def _exact_band(case, q, key):
    n, nb = case["size"], case["bands"]
    d, N, obs = _data(q)
    tau, P = float(N[obs].min()), q["P"].double()
    a, w, sd = _t_terms(d, N, obs, tau)
    bins = q["bins"].long()
    sel = bins.reshape(-1) >= 0
    idx = bins.reshape(-1)[sel]
    weight = torch.full((n, n // 2 + 1), 2.0, dtype=F64, device=DEV)
    weight[:, 0] = weight[:, n // 2] = 1.0
    C = case["chains"]
    chains = list(range(C))
    Pb = q["P0"].double()[None].repeat(C, 1)
    s = torch.zeros(C, n, n, dtype=F64, device=DEV)
    out = torch.empty(C, case["samples"], n, n, dtype=F64, device=DEV)
    outP = torch.empty(C, case["samples"], nb, dtype=F64, device=DEV)
    for i in range(case["samples"] * case["thin"]):
        Pk = torch.where(bins[None] >= 0, Pb[:, bins.clamp(min=0)], P[None])
        t = a + w * s + sd * _xi(n, i, chains, 0, key)
        sh = Pk / (Pk + tau) * _rfft(t) + torch.sqrt(Pk * tau / (Pk + tau)) * _zeta(n, i, chains, 1, key)
        zb = _zeta(n, i, chains, 6, key)
        S = torch.zeros(C, nb, dtype=F64, device=DEV)
        X = torch.zeros(C, nb, dtype=F64, device=DEV)
        S.index_add_(1, idx, (weight * sh.abs() ** 2).reshape(C, -1)[:, sel])
        X.index_add_(1, idx, (weight * zb.abs() ** 2).reshape(C, -1)[:, sel])
        Pb = torch.where(X > 0, S / X.clamp(min=1e-300), torch.zeros_like(S))
        s = _irfft(sh, n)
        if (i + 1) % case["thin"] == 0:
            out[:, (i + 1) // case["thin"] - 1] = s
            outP[:, (i + 1) // case["thin"] - 1] = Pb
    return out, outP


def _exact_shear(case, q, key):
    n, C = case["size"], case["chains"]
    chains = list(range(C))
    obs = q["mask"] == 0
    d, N = (q["d1"].double(), q["d2"].double()), (q["N1"].double(), q["N2"].double())
    tau = min(float(N[0][obs].min()), float(N[1][obs].min()))
    terms = [_t_terms(d[k], N[k], obs, tau) for k in range(2)]
    c, s = _rotation(n)
    P = (q["PE"].double(), q["PB"].double())
    f = [p / (p + tau) for p in P]
    gs = [torch.sqrt(p * tau / (p + tau)) for p in P]
    g = [torch.zeros(C, n, n, dtype=F64, device=DEV) for _ in range(2)]
    out = torch.empty(C, case["samples"], 2, n, n, dtype=F64, device=DEV)
    for i in range(case["samples"] * case["thin"]):
        a, b = [_rfft(terms[k][0] + terms[k][1] * g[k] + terms[k][2] * _xi(n, i, chains, 8 * k, key)) for k in range(2)]
        e = f[0] * (c * a + s * b) + gs[0] * _zeta(n, i, chains, 1, key)
        m = f[1] * (c * b - s * a) + gs[1] * _zeta(n, i, chains, 9, key)
        g = [_irfft(c * e - s * m, n), _irfft(s * e + c * m, n)]
        if (i + 1) % case["thin"] == 0:
            j = (i + 1) // case["thin"] - 1
            out[:, j, 0], out[:, j, 1] = g[0], g[1]
    return out


def _exact_batch(case, seed):
    groups, _ = _batch_images(case, seed)
    res, first = [], 0
    for q in groups:
        n, c = q["size"], q["count"]
        d, N, obs = q["d"].double(), q["N"].double(), q["mask"] == 0
        P = q["P"].double()
        w = torch.empty(c, n, n, dtype=F64, device=DEV)
        for lo in range(0, c, 64):
            sl = slice(lo, lo + 64)
            w[sl] = _cg(_scalar_S(P[sl], n), d[sl], N[sl], obs[sl])[0]
        tau = torch.where(obs, N, torch.full_like(N, math.inf)).amin((1, 2), keepdim=True)
        out = torch.empty(c, case["samples"], n, n, dtype=F64, device=DEV)

        def keep(i, s):
            out[:, i - 1] = s

        _chain(w, _t_terms(d, N, obs, tau), P, tau, n, case["samples"], list(range(first, first + c)), int(seed), keep)
        first += c
        res.append((w, out))
    return res


def _exact_gradient(case, q, key):
    n = case["size"]
    amp, slope, k0, alpha = q["amp"], q["slope"], q["k0"], q["alpha"]
    k = _wavenumber(n)
    k[0, 0] = k0
    P = amp * (k / k0) ** slope
    P[0, 0] = 0.0
    dPs = (P / amp, P * torch.log(k / k0))
    s2, d, obs = q["N"].double(), q["d"].double(), q["mask"] == 0
    N = alpha * s2
    S = _scalar_S(P, n)
    weight = torch.full((n, n // 2 + 1), 2.0, dtype=F64, device=DEV)
    weight[:, 0] = weight[:, n // 2] = 1.0

    def cross(dP, a, b):
        return float((weight * dP * (_rfft(a).conj() * _rfft(b)).real).sum())

    probes = []
    for j in range(case["probes"]):
        w = torch.stack(_philox(*[torch.as_tensor(v, device=DEV, dtype=torch.int64).expand(n * n // 4) for v in
                                  (torch.arange(n * n // 4, device=DEV), j, 0, 5)], key), -1).reshape(n, n)
        probes.append(torch.where(obs, torch.where(w >> 31 != 0, -1.0, 1.0).double(), torch.zeros_like(d)))
    g = q["g"].double()
    rhs = torch.stack([torch.where(obs, d, torch.zeros_like(d))] + probes + [torch.where(obs, S(g), torch.zeros_like(d))])
    sol, x = _cg(S, rhs, N.expand_as(rhs), obs.expand_as(rhs))
    o = obs.double()
    xd, xs = x[0], x[1:-1]
    gq = [0.5 * cross(dP, xd, xd) for dP in dPs] + [0.5 * float((o * s2 * xd * xd).sum())]
    tr = [0.0, 0.0, 0.0]
    for z, cz in zip(probes, xs):
        for i, dP in enumerate(dPs):
            tr[i] += cross(dP, z, cz) / len(probes)
        tr[2] += float((o * s2 * z * cz).sum()) / len(probes)
    y = x[-1]
    vjp = [cross(dP, g - y, xd) for dP in dPs] + [-float((o * s2 * y * xd).sum())]
    as64 = lambda v: torch.tensor(v, dtype=F64)  # noqa: E731
    return (-0.5 * float((d * o * xd).sum()), as64(gq), as64([a - 0.5 * b for a, b in zip(gq, tr)]), sol[0], as64(vjp))

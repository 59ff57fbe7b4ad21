"""CPU checks of the index algebra behind the on-chip kernels with several threads per row (32^2, 64^2 and
128^2), restated in FP64 NumPy:

* a transform of length B A in two in-place passes (B-point DFTs over the A-strided subsequences n0 + A m,
  twiddle W^(n0 q) at position A q + n0, then A-point DFTs of unit q, X[q + B j] at position A q + j), and its
  inverse run backwards;
* the two units of a thread, q and B - q (0 and B/2 for the first), with the first thread's swap, hold every mode
  pair (k, -k) once, in the pair pattern (p[j], q[A-1-j]), (q[j], p[A-1-j]) with the stated frequencies;
* the slot order of the mode tables.
"""
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1810_02821_gb300 import build

SIZES = [32, 64, 128]


def _geo(N):
    A = 8 if N >= 64 else 4
    return A, (N // 2) // A, N // A   # A, row radix BR, column radix BC


def _forward(x, A, B):
    n, buf = x.size, np.array(x, complex)
    for n0 in range(A):
        c = np.fft.fft(buf[n0 + A * np.arange(B)])
        buf[n0 + A * np.arange(B)] = c * np.exp(-2j * np.pi * n0 * np.arange(B) / n)
    for q in range(B):
        buf[A * q:A * q + A] = np.fft.fft(buf[A * q:A * q + A])
    return buf


def _inverse(buf, A, B):
    n, x = buf.size, np.array(buf, complex)
    for q in range(B):
        x[A * q:A * q + A] = np.fft.ifft(x[A * q:A * q + A]) * A * np.exp(2j * np.pi * q * np.arange(A) / n)
    for n0 in range(A):
        x[n0 + A * np.arange(B)] = np.fft.ifft(x[n0 + A * np.arange(B)]) * B
    return x


def _pairs(A, B, h):
    """Frequency pairs of the thread with units (h, hb), in the order the kernels run them."""
    hb = B // 2 if h == 0 else B - h
    p, q = [h + B * j for j in range(A)], [hb + B * j for j in range(A)]
    if h == 0:   # swap of the upper halves, unit 0's rotated
        t = p[A // 2:]
        p = p[:A // 2] + q[A // 2:]
        q = q[:A // 2] + t[1:] + t[:1]
    return [(p[j], q[A - 1 - j], h + B * j) for j in range(A // 2)] + \
           [(q[j], p[A - 1 - j], hb + B * j) for j in range(A // 2)]


@pytest.mark.parametrize("N", SIZES)
def test_two_pass_transform_and_inverse(N):
    A, BR, BC = _geo(N)
    rng = np.random.default_rng(N)
    for n, B in ((N // 2, BR), (N, BC)):
        x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
        buf, X = _forward(x, A, B), np.fft.fft(x)
        k = np.array([s // A + B * (s % A) for s in range(n)])   # frequency held by position s
        assert np.allclose(buf, X[k], atol=1e-10)
        assert np.allclose(_inverse(buf, A, B), n * x, atol=1e-9)


@pytest.mark.parametrize("N", SIZES)
def test_unit_pairs_cover_every_mode_pair_once(N):
    A, BR, BC = _geo(N)
    for n, B in ((N // 2, BR), (N, BC)):
        seen, leads = [], []
        for h in range(B // 2):
            for a, b, lead in _pairs(A, B, h):
                assert a == lead and (b == n - a if a else b == n // 2)
                seen += [a, b]
                leads.append(a)
        assert sorted(seen) == list(range(n))
        assert sorted(leads) == sorted(min(a, (n - a) % n) if a else 0 for a in leads)  # leads below n/2
        assert sorted(leads) == list(range(n // 2))


@pytest.mark.parametrize("N", SIZES)
def test_slot_order_of_the_mode_tables(N):
    A, BR, _ = _geo(N)
    L = N // 2
    for kx in range(L):   # mode_pos with cm = BR
        slot = (kx % BR) * (L // BR) + kx // BR
        assert slot // A + BR * (slot % A) == kx


@pytest.fixture(scope="module")
def kernel_part():
    """part(R, n_chains, n_sweeps, [(i, s), ...]) -> rows (exists, chain, first, end, load, save, polls) from the kernels'
    own share arithmetic, compiled for the host."""
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available to build the host driver")
    tmp = tempfile.mkdtemp()
    exe = os.path.join(tmp, "shares")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "helpers", "shares_host.cu")
    subprocess.run([build.nvcc_path(), *build.ARCH, "-std=c++17", "-o", exe, src], check=True, cwd=tmp, capture_output=True)

    def part(R, n_chains, S, which):
        inp = "".join(f"{R} {n_chains} {S} {i} {s}\n" for i, s in which)
        out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]

    yield part
    shutil.rmtree(tmp, ignore_errors=True)


def _parts(i, R, n_chains, S):
    """Parts (chain, first sweep, end, load, save) of CTA i, in the order it runs them."""
    W = n_chains * S
    q, r = divmod(W, R)
    a, b = q * i + r * i // R, q * (i + 1) + r * (i + 1) // R
    out = []
    if b % S:
        out.append((b // S, 0, b % S, False, True))
    out += [(c, 0, S, False, False) for c in range((a + S - 1) // S, b // S)]
    if a % S:
        out.append((a // S, a % S, S, True, False))
    return out


@pytest.mark.parametrize("R,n_chains,S", [(152, 200, 30), (304, 1000, 7), (304, 305, 1), (5, 6, 100), (7, 13, 3), (3, 3, 4)])
def test_balanced_shares_cover_every_sweep_once_and_hand_over_in_time(kernel_part, R, n_chains, S):
    """Equal shares of all chains' sweeps: every sweep once, at most two parts a chain, the first part of a split chain
    at the start of its CTA and the second at the end of the next one, one sweep before the first has finished at the
    earliest. The kernels' own parts (kpart_of, compiled for the host) are the ones checked here."""
    parts = [_parts(i, R, n_chains, S) for i in range(R)]
    got = iter(kernel_part(R, n_chains, S, [(i, s) for i in range(R) for s in range(len(parts[i]) + 1)]))
    for own in parts:
        assert [row[:6] for row in (next(got) for _ in own)] == [(1, c, d0, d1, int(load), int(save)) for c, d0, d1, load, save in own]
        assert next(got)[0] == 0   # and no further part
    seen, loads, length = {}, {}, []
    for i in range(R):
        t = 0
        for k, (c, d0, d1, load, save) in enumerate(parts[i]):
            assert d0 < d1
            seen.setdefault(c, []).append((d0, d1))
            if save:
                assert k == 0
                loads.setdefault(c, {})["ready"] = (i, d1)
            if load:
                loads.setdefault(c, {})["start"] = (i, t)
            t += d1 - d0
        length.append(t)
    for c in range(n_chains):
        spans = sorted(seen[c])
        assert len(spans) <= 2 and spans[0][0] == 0 and spans[-1][1] == S and all(x[1] == y[0] for x, y in zip(spans, spans[1:]))
    for c, v in loads.items():
        assert v["start"][0] == v["ready"][0] + 1 and v["start"][1] >= v["ready"][1] - 1   # equal shares to one sweep
    assert max(length) - min(length) <= 1


@pytest.mark.parametrize("R,n_chains,S", [(304, 2 ** 31 - 1, 2 ** 31 - 1), (760, 2 ** 31 - 5, 2 ** 31 - 1), (152, 2 ** 31 - 1, 2 ** 30)])
def test_share_arithmetic_near_the_largest_sweep_count(kernel_part, R, n_chains, S):
    """n_chains n_sweeps close to 2^62: the first and last parts of each share, in exact integers."""
    W = n_chains * S
    q, r = divmod(W, R)
    for i in (0, 1, 2, R // 2, R - 2, R - 1):
        a, b = q * i + r * i // R, q * (i + 1) + r * (i + 1) // R
        head = int(b % S > 0)
        whole = b // S - (a + S - 1) // S
        rows = kernel_part(R, n_chains, S, [(i, s) for s in (0, head, head + whole - 1, head + whole, head + whole + 1)])
        if head:
            assert rows[0][:6] == (1, b // S, 0, b % S, 0, 1)
        assert rows[1][:6] == (1, (a + S - 1) // S, 0, S, 0, 0) and rows[2][:6] == (1, b // S - 1, 0, S, 0, 0)
        if a % S:
            assert rows[3][:6] == (1, a // S, a % S, S, 1, 0)
        assert rows[3][0] == int(a % S > 0) and rows[4][0] == 0


@pytest.mark.parametrize("R,n_chains,S", [(304, 305, 7), (304, 305, 10 ** 7), (152, 200, 2 ** 31 - 1)])
def test_the_wait_for_a_state_outlasts_its_sweeps(kernel_part, R, n_chains, S):
    """A CTA may come to the rest of a chain a sweep before the state is ready, and its pace over that part may differ from
    the other CTA's: the limit of the wait, at 0.3 us a poll or more, is a second and then 0.1 ms for every sweep waited for."""
    for row in kernel_part(R, n_chains, S, [(i, s) for i in range(R) for s in range(4)]):
        exists, _, first, _, load, _, polls = row
        if exists and load:
            assert polls * 0.3e-6 >= 1.0 + 0.1e-3 * first

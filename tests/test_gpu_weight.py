"""The Wiener filters' pixel weight 1 / (1 + lt inb) on the device (approximate reciprocal and one Newton-Raphson step)
over its whole range, against FP64."""
import os
import subprocess

import numpy as np
import pytest

from gpu_common import need_gpu
from paper_1810_02821_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def weight(tmp_path_factory):
    need_gpu()
    exe = str(tmp_path_factory.mktemp("weight") / "weight")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "helpers", "weight_device.cu")
    subprocess.run([build.nvcc_path(), *build.ARCH, *build.FLAGS, "-o", exe, src], check=True, capture_output=True)

    def run(lt, inb):
        inp = "".join(f"{float(a).hex() if np.isfinite(a) else 'inf'} {float(b).hex() if np.isfinite(b) else 'inf'}\n"
                      for a, b in zip(lt, inb))
        out = subprocess.run([exe], input=inp, capture_output=True, text=True, check=True).stdout
        return np.array([float.fromhex(x) for x in out.split()])

    return run


def test_weight_within_an_ulp(weight):
    """Relative to the exact weight: half an ulp from 1 + lt inb rounded to FP32 and half an ulp from the result, each 2^-24
    of its value at most, and what the Newton step leaves of the reciprocal's ulp, its square; lt inb up to 2^125, above
    which the reciprocal is flushed to zero."""
    rng = np.random.default_rng(1)
    lt = np.float32(2.0) ** rng.uniform(-60, 60, 40000).astype(np.float32)
    inb = (2.0 ** rng.uniform(-40, 65, 40000)).astype(np.float32)
    exact = 1.0 / (1.0 + lt.astype(np.float64) * inb.astype(np.float64))
    err = np.abs(weight(lt, inb) - exact) / exact
    print(f"largest relative error {err.max():.3e}, {err.max() * 2 ** 24:.3f} times 2^-24")
    assert err.max() <= 2.05 * 2.0 ** -24


def test_weight_at_the_ends(weight):
    lt = np.array([1.0, 1e30, 1e-30, 1.0, 1e10, 1e30], np.float32)
    inb = np.array([0.0, 0.0, 0.0, np.inf, np.inf, 1e30], np.float32)   # exact data; no noise left; overflow
    assert list(weight(lt, inb)) == [1.0, 1.0, 1.0, 0.0, 0.0, 0.0]
    far = weight(np.full(3, 2.0 ** 100, np.float32), np.float32([2.0 ** 25.5, 2.0 ** 26, 2.0 ** 27]))
    assert np.all((far >= 0.0) & (far <= 2.0 ** -125))   # subnormal weights are flushed

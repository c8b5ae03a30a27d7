"""The error of one free-space step of metres, whose increment is as large as the
field: it carries every rounded constant of the two transforms in full.

Random fields of one row, so that every mode counts, against the oracle's
propagator in FP64.  Bound per size: the relative error of the kernels of 16
points per thread on the same fields (measured), whose transforms have the fewest
passes, and 5 % for the roundings falling otherwise.  With twiddles rounded to
one float each the error was 1.02 (N = 4096) to 1.42 times (N = 128) that."""

import cmath
import math

import numpy as np
import pytest

from oracle import run as orun
from paper_2601_06340_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

ERROR_16 = {64: 1.203e-7, 128: 1.306e-7, 256: 1.945e-7, 512: 2.097e-7, 1024: 2.207e-7,
            2048: 2.307e-7, 4096: 2.498e-7, 8192: 2.513e-7, 16384: 2.505e-7}


@pytest.mark.parametrize("nx", sorted(ERROR_16))
def test_far_field_error(bpm_lib, monkeypatch, nx):
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    wl = inputs.far_field_step(np.zeros((1, 2, nx)), nx, 0.1, -0.05 * nx, 2.0e6)
    p = orun.plans_for(wl)[0]
    prop = np.stack([p.prop_plus, p.prop_minus])
    g = cmath.exp(1j * math.fmod(math.fmod(p.dzh * p.c, 2.0 * math.pi), 2.0 * math.pi))
    num = den = 0.0
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:
        for seed in range(max(2, 65536 // nx)):
            rng = np.random.default_rng(seed)
            f = rng.standard_normal((1, 2, nx)) + 1j * rng.standard_normal((1, 2, nx))
            f = f.astype(np.complex64).astype(np.complex128)
            out = plan.propagate(f, records=False, powers=False).psi[0]
            ref = np.fft.ifft(np.fft.fft(f[0]) * prop) * g
            num += np.sum(np.abs(out - ref) ** 2)
            den += np.sum(np.abs(ref) ** 2)
    err = math.sqrt(num / den)
    print(f"nx={nx}: {err:.4g}, {err / ERROR_16[nx]:.3f} of the 16-point kernels'")
    assert err <= 1.05 * ERROR_16[nx], err

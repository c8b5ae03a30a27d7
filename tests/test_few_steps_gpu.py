"""First-order launches of up to four steps on the 8-points-per-thread kernels, which
apply every twiddle with its low part (kFewSteps): every size and cluster size, on
random two-band fields through a masked, strained crystal, a record and its band
powers at every step, one launch of four steps or a step and three, against the
FP64 oracle.

Tolerance per step: the field's sum with the increment and the coupling round five
times (5 * 2^-24 = 3e-7), the two transforms of the increment, which is at most as
large as the field, by 0.6 * 2^-24 * sqrt(2 log2 nx) <= 1.9e-7; 5e-7 a step.
"""

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs
from parity_util import band_errors, run_ref

pytestmark = pytest.mark.gpu

CASES = [(64, 1), (64, 33), (128, 5), (256, 1), (512, 101), (1024, 1), (1024, 151), (2048, 1),
         (2048, 30), (4096, 1), (4096, 36), (8192, 1), (8192, 15), (16384, 1), (16384, 7)]


@pytest.mark.parametrize("parts", [(0, 4), (0, 1, 4)])
@pytest.mark.parametrize("nx,rows", CASES)
def test_few_steps_match_oracle(bpm_lib, monkeypatch, nx, rows, parts):
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    rng = np.random.default_rng(nx + rows)
    wl = inputs.pulse_batched(nx=nx, nz=4, n_energy=rows, dx_um=0.4, record_every=1)
    wl.psi0 = rng.standard_normal((rows, 2, nx)) + 1j * rng.standard_normal((rows, 2, nx))
    wl.crystal = dict(kind=inputs.CRYSTAL_MASK, mask=(rng.uniform(size=(4, nx)) < 0.8))
    wl.strain = dict(kind=inputs.STRAIN_ARRAY, ux=rng.uniform(-1e-3, 1e-3, (4, nx)))
    pick = sorted({0, rows // 2, rows - 1})
    ref = run_ref(wl, rows=pick)
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:
        psi = wl.psi0
        for a, b in zip(parts, parts[1:]):
            out = plan.propagate(psi, a, b)
            assert binding.bpm_launch_ctas(plan.handle) > 0
            psi = out.psi
            for n in range(a, b):
                errs = band_errors(out.records[pick][:, n], ref.records[:, n])
                assert max(errs) <= 5e-7 * (n + 1), (n, errs)
            assert np.allclose(out.powers[pick][:, a:b], ref.powers[:, a:b], rtol=1e-5)
    assert max(band_errors(psi[pick], ref.psi)) <= 5e-7 * 4

"""The grid barrier of the FP64 and 3D marches gives up without a fault.

The self-test kernel's counter is one arrival short, so its first wait runs to a
limit of some 4 ms (16384 polls) and the kernel, like a march, goes on without
waiting again and sets the status bit that the host turns into BPM_ERR_TIMEOUT.
An FP64 and a 3D march on the same context afterwards equal the oracle."""

import pytest

from oracle import run as orun
from paper_2601_06340_gb300 import binding, inputs

from parity_util import TOL_FP32, TOL_FP64, band_errors, run_ref

pytestmark = pytest.mark.gpu


def test_expired_barrier_sets_status_and_context_stays_usable(bpm_lib):
    status, seconds = binding.bpm_selftest_barrier_expiry()
    assert status == 1
    assert 0.0 < seconds < 1.0, seconds
    print(f"barrier gave up after {1e3 * seconds:.2f} ms")
    wl = inputs.laue_perfect(nx=1024, nz=60, record_every=20)
    with binding.Plan(wl, binding.BPM_FP64_PLAIN) as plan:
        out = plan.propagate()
        assert binding.bpm_device_status(plan.handle) == binding.BPM_OK
    ref = run_ref(wl)
    assert max(band_errors(out.psi, ref.psi, out.records, ref.records)) <= TOL_FP64
    wl = inputs.cube_dislocation_3d(nx=256, ny=256, nz=6, dx_um=0.08, dy_um=0.08, dz_um=0.1,
                                    cube_um=5.0, fwhm_um=1.5)
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:
        out = plan.propagate(records=False)
    assert max(band_errors(out.psi, orun.run_workload3d(wl).psi)) <= TOL_FP32

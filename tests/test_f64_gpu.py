"""The FP64 march in one launch (csrc/f64_kernel.cuh), nx = 64 .. 16384.

Random two-band fields (every mode and cell carries weight) through a masked,
strained crystal with a ragged record tail against the FP64 oracle: every
size with one row (a few CTAs) and with row counts that give a CTA several
items per phase, all three splittings.  nx = 32 marches pass by pass.

Tolerance: a step rounds a value in each of 2 log2(nx) butterflies, the
propagator and the coupling (at most 2 * 14 + 8 roundings of 2^-53); over 40
steps that is below 1.6e-13 for either side if every rounding pushes the same
way, so 3.2e-13 between them, and three times the propagations for Forest-Ruth.
"""

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs
from parity_util import band_errors, run_ref

pytestmark = pytest.mark.gpu

FIRST, VERLET, FR = (binding.BPM_SPLIT_FIRST_ORDER, binding.BPM_SPLIT_VERLET,
                     binding.BPM_SPLIT_FOREST_RUTH)
METHOD = {FIRST: "first_order", VERLET: "verlet", FR: "forest_ruth"}
NZ, EVERY = 40, 7


def _workload(nx, rows):
    rng = np.random.default_rng(nx + rows)
    wl = inputs.pulse_batched(nx=nx, nz=NZ, n_energy=rows, dx_um=0.4, record_every=EVERY)
    wl.psi0 = rng.standard_normal((rows, 2, nx)) + 1j * rng.standard_normal((rows, 2, nx))
    wl.crystal = dict(kind=inputs.CRYSTAL_MASK, mask=(rng.uniform(size=(NZ, nx)) < 0.8))
    wl.strain = dict(kind=inputs.STRAIN_ARRAY, ux=rng.uniform(-1e-3, 1e-3, (NZ, nx)))
    return wl


CASES = [(nx, 1) for nx in (32, 64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384)]
CASES += [(64, 3000), (512, 301), (4096, 37), (16384, 11)]


@pytest.mark.parametrize("split", [FIRST, VERLET, FR])
@pytest.mark.parametrize("nx,rows", CASES)
def test_fp64_matches_oracle(bpm_lib, nx, rows, split):
    wl = _workload(nx, rows)
    with binding.Plan(wl, binding.BPM_FP64_PLAIN, splitting=split) as plan:
        out = plan.propagate()
        first = plan.propagate(n_end=17, records=False, powers=False)
        rest = plan.propagate(psi_in=first.psi, n_begin=17, records=False, powers=False)
    pick = sorted({0, rows // 2, rows - 1})
    ref = run_ref(wl, method=METHOD[split], rows=pick)
    tol = 9.6e-13 if split == FR else 3.2e-13
    errs = band_errors(out.psi[pick], ref.psi, out.records[pick], ref.records)
    assert max(errs) <= tol, errs
    assert max(band_errors(rest.psi[pick], ref.psi)) <= tol
    assert np.allclose(out.powers[pick], ref.powers, rtol=2 * tol, atol=0)


def test_fp64_request_equals_the_solve_alone(bpm_lib):
    """The server marches FP64 requests in epochs of the same kernel, beside
    FP32 ones."""
    binding.bpm_server_configure(0.6, 64, 16, 1000)
    wls = [_workload(1024, 1), _workload(2048, 3), _workload(512, 1)]
    precs = [binding.BPM_FP64_PLAIN, binding.BPM_FP64_PLAIN, binding.BPM_FP32_FUSED]
    plans = [binding.Plan(wl, p) for wl, p in zip(wls, precs)]
    outs = [np.empty_like(wl.psi0) for wl in wls]
    try:
        tickets = [binding.bpm_submit(p.handle, wl.psi0, o)
                   for p, wl, o in zip(plans, wls, outs)]
        for t in tickets:
            assert binding.bpm_poll(t, -1) == binding.BPM_OK
        for p, wl, o, prec in zip(plans, wls, outs, precs):
            alone = p.propagate(records=False, powers=False).psi
            errs = band_errors(o, alone)
            assert max(errs) <= (1e-15 if prec == binding.BPM_FP64_PLAIN else 2e-4), errs
    finally:
        for p in plans:
            p.close()
        binding.bpm_server_configure(0.6, 256, 256, 100000)

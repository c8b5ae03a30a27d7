"""Rows of 8 points per thread: spread over clusters of 8 or 16 CTAs
(csrc/spread_kernel.cuh) or one row per CTA (csrc/row_kernel.cuh).

Every size and cluster size of the form, on random two-band fields (every
mode and cell carries weight) through a masked, strained crystal stored as a
per-cell stream, with a ragged record tail, against the FP64 oracle row by
row: single rows and the row counts where the rule changes the cluster size
or runs a second wave.  The separable slices, full-size marches, resumed
marches, graph capture and repeat runs of the form are covered by the tests
of those features, which take it by default.

Tolerance: one step rounds the field once (relative error <= 2^-24 per
component) and the per-step increment, which is at most the field's size,
with the FFT's error of a few 2^-24 per pass; over 40 steps of random walk
that is below 40 * 2^-24 = 2.4e-6 for the first-order step, three times the
propagations for Forest-Ruth.
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


def _workload(nx, rows, nz=NZ):
    rng = np.random.default_rng(nx + rows)
    wl = inputs.pulse_batched(nx=nx, nz=nz, n_energy=rows, dx_um=0.4, record_every=EVERY)
    wl.psi0 = rng.standard_normal((rows, 2, nx)) + 1j * rng.standard_normal((rows, 2, nx))
    wl.crystal = dict(kind=inputs.CRYSTAL_MASK, mask=(rng.uniform(size=(nz, nx)) < 0.8))
    wl.strain = dict(kind=inputs.STRAIN_ARRAY, ux=rng.uniform(-1e-3, 1e-3, (nz, nx)))
    return wl


# (nx, rows): one row, then the counts at which the rule changes
CASES = [(64, 1), (64, 33), (128, 1), (256, 5), (512, 1), (512, 101), (1024, 1), (1024, 77),
         (1024, 151), (2048, 1), (2048, 7), (2048, 8),
         (4096, 1), (4096, 33), (8192, 1), (8192, 15), (8192, 17), (16384, 1), (16384, 8)]


@pytest.mark.parametrize("split", [FIRST, VERLET, FR])
@pytest.mark.parametrize("nx,rows", CASES)
def test_spread_matches_oracle(bpm_lib, monkeypatch, nx, rows, split):
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    wl = _workload(nx, rows)
    with binding.Plan(wl, binding.BPM_FP32_FUSED, splitting=split) as plan:
        out = plan.propagate()
    pick = sorted({0, rows // 2, rows - 1})
    ref = run_ref(wl, method=METHOD[split], rows=pick)
    tol = 7.2e-6 if split == FR else 2.4e-6
    errs = band_errors(out.psi[pick], ref.psi, out.records[pick], ref.records)
    assert max(errs) <= tol, errs
    assert np.allclose(out.powers[pick], ref.powers, rtol=1e-5)


@pytest.mark.parametrize("split", [FIRST, VERLET, FR])
@pytest.mark.parametrize("nx,rows", [(2048, 90), (4096, 45), (8192, 17), (16384, 8)])
def test_rotating_rows_match_oracle(bpm_lib, monkeypatch, nx, rows, split):
    """More rows than a launch keeps resident, in chunks with a shorter last
    one: 151 steps, so twice the bound of 40 (random walk)."""
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    wl = _workload(nx, rows, 151)
    with binding.Plan(wl, binding.BPM_FP32_FUSED, splitting=split) as plan:
        out = plan.propagate()
        assert 0 < binding.bpm_launch_shape(plan.handle)[1] < 151
    pick = [0, rows - 1]
    ref = run_ref(wl, method=METHOD[split], rows=pick)
    tol = 14.4e-6 if split == FR else 4.8e-6
    errs = band_errors(out.psi[pick], ref.psi, out.records[pick], ref.records)
    assert max(errs) <= tol, errs
    assert np.allclose(out.powers[pick], ref.powers, rtol=1e-5)

"""Which kernels rows march on, and the kernels that the rule no longer takes alone.

By default single rows of nx >= 64 march with 8 points per thread, which
bpm_launch_ctas tells apart; with BPM_FUSED_LAYOUT set they take the kernels of 16
points per thread (and the half-band split), which batches, the server's splitting
requests and that variable still run.  Those against the FP64 oracle, on random
two-band fields through a masked, strained crystal (per-cell stream) and through a
bent one (separable slices), with a ragged record tail.

Tolerance: as in test_spread_gpu.py, 40 steps of one rounding of the field each
(40 * 2^-24 = 2.4e-6), three times that for Forest-Ruth's propagations; rows of nx
<= 128 propagate the whole field here, with a transform pair's rounding of 0.6 *
2^-24 * sqrt(2 log2 nx) = 1.34e-7 a step: 40 of them, 5.4e-6.
"""

import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs
from parity_util import band_errors, run_ref

pytestmark = pytest.mark.gpu

FIRST, VERLET, FR = (binding.BPM_SPLIT_FIRST_ORDER, binding.BPM_SPLIT_VERLET,
                     binding.BPM_SPLIT_FOREST_RUTH)
METHOD = {FIRST: "first_order", VERLET: "verlet", FR: "forest_ruth"}


def _workload(nx, form, nz=40):
    rng = np.random.default_rng(nx)
    if form == "stream":
        wl = inputs.pulse_batched(nx=nx, nz=nz, n_energy=1, dx_um=0.4, record_every=7)
        wl.crystal = dict(kind=inputs.CRYSTAL_MASK, mask=(rng.uniform(size=(nz, nx)) < 0.8))
        wl.strain = dict(kind=inputs.STRAIN_ARRAY, ux=rng.uniform(-1e-3, 1e-3, (nz, nx)))
    else:
        wl = inputs.bragg_bent(nx=nx, nz=nz, record_every=7)
    wl.psi0 = rng.standard_normal((1, 2, nx)) + 1j * rng.standard_normal((1, 2, nx))
    return wl


@pytest.mark.parametrize("nx,rows,ctas", [
    (32, 1, 0), (64, 1, 1), (256, 40, 1), (512, 1, 1), (1024, 1, 8), (1024, 150, 1), (2048, 1, 16),
    (2048, 30, 8), (2048, 140, 0), (4096, 1, 16), (4096, 90, 0), (8192, 1, 16), (16384, 1, 16)])
def test_rule(bpm_lib, monkeypatch, nx, rows, ctas):
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    wl = inputs.pulse_batched(nx=nx, nz=6, n_energy=rows, dx_um=0.4)
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:
        assert binding.bpm_launch_ctas(plan.handle) == 0
        plan.propagate(records=False)
        assert binding.bpm_launch_ctas(plan.handle) == ctas
        monkeypatch.setenv("BPM_FUSED_LAYOUT", "split")
        plan.propagate(records=False)
        assert binding.bpm_launch_ctas(plan.handle) == 0


@pytest.mark.parametrize("form", ["stream", "separable"])
@pytest.mark.parametrize("split,sizes", [(FIRST, {64: -1, 512: -1, 1024: -1, 2048: -1, 4096: 2,
                                                  8192: -1, 16384: -1}),
                                         (VERLET, {128: 3, 512: 4, 1024: 4, 2048: 3, 4096: 5,
                                                   8192: 5, 16384: 5}),
                                         (FR, {64: 6, 512: 10, 1024: 10, 2048: 10, 4096: 9,
                                               8192: 9})])
def test_former_kernels_match_oracle(bpm_lib, monkeypatch, form, split, sizes):
    monkeypatch.setenv("BPM_FUSED_LAYOUT", "split")
    monkeypatch.setenv("BPM_SLICE_STREAM", "1" if form == "stream" else "0")
    for nx, layout in sizes.items():
        wl = _workload(nx, form)
        with binding.Plan(wl, binding.BPM_FP32_FUSED, splitting=split) as plan:
            out = plan.propagate()
            assert binding.bpm_launch_shape(plan.handle)[0] == layout, nx
            assert binding.bpm_launch_ctas(plan.handle) == 0
            assert binding.bpm_slice_form(plan.handle)[0] == (form == "separable")
        ref = run_ref(wl, method=METHOD[split])
        tol = (5.4e-6 if nx <= 128 else 2.4e-6) * (3 if split == FR else 1)
        errs = band_errors(out.psi, ref.psi, out.records, ref.records)
        assert max(errs) <= tol, (nx, errs)
        assert np.allclose(out.powers, ref.powers, rtol=1e-5), nx


def test_plain_constants_keep_their_kernels(bpm_lib):
    """BPM_FUSED_EXACT=0 (read once in a process) asks for plain butterfly constants,
    which only the kernels of 16 points per thread and the half-band split have."""
    code = """
import os
os.environ.pop("BPM_FUSED_LAYOUT", None)
from paper_2601_06340_gb300 import binding, inputs
with binding.Plan(inputs.bragg_bent(nx=1024, nz=8, record_every=0)) as plan:
    plan.propagate(records=False)
    print(binding.bpm_launch_ctas(plan.handle))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for exact, ctas in (("0", "0"), ("1", "8")):
        out = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True,
                             env=dict(os.environ, BPM_FUSED_EXACT=exact), timeout=300)
        assert out.returncode == 0 and out.stdout.split() == [ctas], (exact, out)

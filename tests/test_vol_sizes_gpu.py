"""The 3D march (csrc/vol_kernel.cuh) at every combination of passes and CTA
shapes, on random two-band fields (every mode and cell carries weight), rows
of two photon energies, against the 3D oracle: lines and tiles per CTA from 1
to 8 (512 x 256 against 256 x 1024), one item per CTA and several (4096 x 256
with two rows), first-order and Verlet steps.

Tolerance: a step rounds the field once and the coupling's four terms into it
(5 * 2^-24 per component at most), the increment's transforms add log2(nx ny)
roundings of its own size; over 4 steps below 1.2e-6 plus 4 * 24 * 6e-8 / 4
(random signs): 3e-6.
"""

import numpy as np
import pytest

from oracle import run as orun
from paper_2601_06340_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

FIRST, VERLET = binding.BPM_SPLIT_FIRST_ORDER, binding.BPM_SPLIT_VERLET
CASES = [(256, 256, 1, FIRST), (256, 1024, 1, FIRST), (512, 512, 2, FIRST), (512, 256, 1, VERLET),
         (1024, 256, 2, FIRST), (2048, 256, 1, FIRST), (4096, 256, 2, FIRST),
         (4096, 256, 1, VERLET), (256, 512, 3, VERLET)]


@pytest.mark.parametrize("nx,ny,rows,split", CASES)
def test_vol_shapes_match_oracle(bpm_lib, nx, ny, rows, split):
    nz = 4
    rng = np.random.default_rng(nx + ny + rows)
    wl = inputs.cube_dislocation_3d(nx=nx, ny=ny, nz=nz, record_every=2, cube_um=0.03 * nx)
    wl.energies_ev = inputs.E_440_EV + 2.0 * np.arange(rows)
    wl.psi0 = (rng.standard_normal((rows, 2, ny, nx)) + 1j * rng.standard_normal((rows, 2, ny, nx)))
    wl.crystal["box_um"] = [0.0, 0.03 * nx, -0.01 * ny, 0.01 * ny, -1.0, 1.0]
    ref = orun.run_workload3d(wl, method="verlet" if split == VERLET else "first_order")
    with binding.Plan(wl, binding.BPM_FP32_FUSED, splitting=split) as plan:
        out = plan.propagate()
    for r in range(rows):
        for b in range(2):
            for got, want in [(out.psi[r, b], ref.psi[r, b])] + [
                    (out.records[r, k, b], ref.records[r, k, b]) for k in range(2)]:
                err = np.linalg.norm(got - want) / np.linalg.norm(want)
                assert err <= 3e-6, (r, b, err)
    assert np.allclose(out.powers, ref.powers, rtol=1e-5)

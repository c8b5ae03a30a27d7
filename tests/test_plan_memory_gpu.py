"""A plan that cannot be made gives back what it had allocated.

Rows of nx = 16384 beyond one launch carry a launch schedule, allocated before
the state and the host staging.  With more rows than the GPU's memory holds,
plan creation runs out in one of those and must return the memory of the
schedule too (24 descriptors a row: hundreds of megabytes here)."""

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

# device bytes per row of 16384 points: the split band's tables (2 MB), the
# natural-order tables and the state (256 KB each); then the staging (512 KB)
TABLES, STAGING = (2048 + 256 + 256) << 10, 512 << 10


def test_failed_plan_leaves_no_memory_behind(bpm_lib):
    torch = pytest.importorskip("torch")
    wl = inputs.serving_request(np.random.default_rng(2), 16384, 4)
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:     # (loads the kernels)
        plan.propagate()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    rows = int(0.95 * free / TABLES)
    assert rows * (TABLES + STAGING) > free
    wl.energies_ev = np.full(rows, wl.energies_ev[0])
    for _ in range(2):
        with pytest.raises(binding.BpmError) as err:
            binding.Plan(wl, binding.BPM_FP32_FUSED)
        assert err.value.code == binding.BPM_ERR_OOM
    assert torch.cuda.mem_get_info()[0] >= free - (32 << 20)

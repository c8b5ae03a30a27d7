"""Energy -> time synthesis (csrc/omega_to_t.cu) at every number of energies
it takes, with line counts below, at and beyond a block's tile, against the oracle.

Tolerance: per line (one x of one band) in the 2-norm, in which the
transform is a multiple of a unitary map.  A radix-2 stage rounds the sum (1
eps) and multiplies by a rounded root (rounding of root and products: 3 eps
at most), eps = 2^-24 or 2^-53, so B energies give 4 log2(B) eps; the input's
rounding to FP32 adds one eps, the oracle's own FP64 error as much again.
"""
import numpy as np
import pytest

from oracle import timeaxis
from paper_2601_06340_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [binding.BPM_FP32_FUSED, binding.BPM_FP64_PLAIN])
@pytest.mark.parametrize("logb", range(1, 13))
def test_every_energy_count(bpm_lib, logb, prec):
    torch = pytest.importorskip("torch")
    nb = 1 << logb
    fp32 = prec == binding.BPM_FP32_FUSED
    rng = np.random.default_rng(logb)
    stream = torch.cuda.current_stream().cuda_stream
    eps = 2.0 ** -24 if fp32 else 2.0 ** -53
    tol = 2 * 4 * logb * eps + eps
    for nx in (1, 7, 16, 33, 300) if logb < 9 else (1, 7, 16, 33):
        f = rng.standard_normal((nb, 2, nx)) + 1j * rng.standard_normal((nb, 2, nx))
        ref = timeaxis.omega_to_t(f)
        dt = torch.complex64 if fp32 else torch.complex128
        x = torch.from_numpy(f).to(dtype=dt, device="cuda:0").contiguous()
        y = torch.full((2, nx, nb), float("nan"), dtype=dt, device="cuda:0")
        binding.bpm_omega_to_t_device(x, y, nb, nx, prec, stream)
        torch.cuda.synchronize()
        err = np.linalg.norm(y.cpu().numpy() - ref, axis=-1)
        assert np.all(err <= tol * np.linalg.norm(ref, axis=-1)), (nx, err.max())

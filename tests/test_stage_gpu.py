"""The start of a device-API march (input, phase factors, row descriptors).

Few rows travel with one launch's parameters, more by copies; an input may be
the output buffer itself, and a buffer of any alignment.  Every form gives
the bits of the host-API march of the same field (the input is exact in
FP32), FP32 and FP64, 2D and 3D."""

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs

pytestmark = pytest.mark.gpu

FP32, FP64 = binding.BPM_FP32_FUSED, binding.BPM_FP64_PLAIN


def _case(name):
    if name == "3d":
        return inputs.cube_dislocation_3d(nx=256, ny=256, nz=4), FP32
    rows, nx, prec = name
    return inputs.pulse_batched(nx=nx, nz=12, n_energy=rows, dx_um=0.4), prec


@pytest.mark.parametrize("name", [(1, 512, FP32), (24, 256, FP32), (25, 256, FP32),
                                  (26, 1024, FP32), (300, 64, FP32), (1, 64, FP64),
                                  (26, 256, FP64), (2, 32, FP64), "3d"],
                         ids=str)
def test_device_march_equals_host_march(bpm_lib, name):
    torch = pytest.importorskip("torch")
    wl, prec = _case(name)
    dtype = torch.complex64 if prec == FP32 else torch.complex128
    size = 8 if prec == FP32 else 16
    wl.psi0 = wl.psi0.astype(np.complex64).astype(np.complex128)
    x = torch.from_numpy(wl.psi0).to("cuda").to(dtype)
    st = torch.cuda.current_stream().cuda_stream
    with binding.Plan(wl, prec) as plan:
        want = plan.propagate(records=False).psi
        got = []
        y = torch.empty_like(x)
        pw = torch.zeros((wl.batch, plan.n_rec + 1, 2), dtype=torch.float64, device="cuda")
        binding.bpm_propagate_device(plan.handle, x, y, None, pw, 0, wl.nz, st)
        got.append(y)
        z = x.clone()                       # in place
        binding.bpm_propagate_device(plan.handle, z, z, None, None, 0, wl.nz, st)
        got.append(z)
        raw = torch.empty(x.numel() * size + 16, dtype=torch.uint8, device="cuda")
        off = raw[4:4 + x.numel() * size]   # four bytes off the type's alignment
        off.copy_(x.reshape(-1).view(torch.uint8))
        w = torch.empty_like(x)
        binding.bpm_propagate_device(plan.handle, off, w, None, None, 0, wl.nz, st)
        got.append(w)
        torch.cuda.synchronize()
        assert binding.bpm_device_status(plan.handle, st) == binding.BPM_OK
    for g in got:
        assert np.array_equal(g.cpu().numpy(), want.astype(g.cpu().numpy().dtype))
    total = np.sum(np.abs(want) ** 2, axis=tuple(range(2, want.ndim)))
    area = wl.dx_um * (wl.dy_um if name == "3d" else 1.0)
    assert np.allclose(pw[:, -1].cpu().numpy(), total * area, rtol=1e-5 if prec == FP32 else 1e-12)

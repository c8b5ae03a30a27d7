"""A served request beside an asynchronous device march of the same plan.

bpm_submit looks at the plan's pending tickets, not at device marches that the
caller has enqueued, and its own streams cannot be ordered with the caller's.
An FP32 request therefore writes memory of its own only; the final band
powers, which blocks of a line sum through scratch memory, must come out on
both sides as they do alone.  Sums run in a fixed order: equal bits."""

import numpy as np
import pytest

from paper_2601_06340_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,rows,nz", [(2048, 3, 64), (4096, 2, 200), (4096, 40, 30)])
def test_final_powers_of_a_request_and_a_device_march(bpm_lib, nx, rows, nz):
    torch = pytest.importorskip("torch")
    binding.bpm_server_configure(0.6, 64, 256, 1000)
    wl = inputs.pulse_batched(nx=nx, nz=nz, n_energy=rows, dx_um=0.1)
    st = torch.cuda.Stream()
    with binding.Plan(wl, binding.BPM_FP32_FUSED) as plan:
        x = torch.from_numpy(wl.psi0.astype(np.complex64)).to("cuda:0")
        y, pw = torch.empty_like(x), torch.zeros((rows, 1, 2), dtype=torch.float64, device="cuda:0")
        torch.cuda.synchronize()

        def device():
            binding.bpm_propagate_device(plan.handle, x, y, None, pw, 0, nz, st.cuda_stream)

        def submit():
            out, p = np.empty_like(wl.psi0), np.zeros((rows, 1, 2))
            return binding.bpm_submit(plan.handle, wl.psi0, out, None, p), out, p

        device()
        st.synchronize()
        dev_alone, field_alone = pw.cpu().numpy(), y.cpu().numpy()
        t, out_alone, srv_alone = submit()
        assert binding.bpm_poll(t, -1) == binding.BPM_OK
        assert np.all(dev_alone > 0) and np.all(srv_alone > 0)
        for _ in range(8):
            pw.zero_()
            torch.cuda.synchronize()
            for _ in range(3):
                device()
            t, out, p = submit()
            assert binding.bpm_poll(t, -1) == binding.BPM_OK
            st.synchronize()
            assert np.array_equal(pw.cpu().numpy(), dev_alone)
            assert np.array_equal(y.cpu().numpy(), field_alone)
            assert np.array_equal(p, srv_alone) and np.array_equal(out, out_alone)


def test_spread_rows_beside_another_splitting(bpm_lib, monkeypatch):
    """More first-order requests of 8192 than the spread kernel keeps resident (14)
    share their bucket with Forest-Ruth ones, which march apart and are not counted
    against that: every request equals its march alone, whatever kernels the two
    took: 20 steps of Forest-Ruth's three propagations on either side, one rounding
    each (2 * 60 * 2^-24 = 7.2e-6)."""
    monkeypatch.delenv("BPM_FUSED_LAYOUT", raising=False)
    binding.bpm_server_configure(0.6, 64, 8, 1000)
    rng = np.random.default_rng(8)
    items = []
    for i in range(22):
        wl = inputs.serving_request(rng, 8192, 20)
        split = binding.BPM_SPLIT_FOREST_RUTH if i % 4 == 3 else binding.BPM_SPLIT_FIRST_ORDER
        plan = binding.Plan(wl, binding.BPM_FP32_FUSED, splitting=split)
        items.append((plan, wl, np.empty_like(wl.psi0)))
    tickets = [binding.bpm_submit(plan.handle, wl.psi0, out) for plan, wl, out in items]
    for t in tickets:
        assert binding.bpm_poll(t, -1) == binding.BPM_OK
    binding.bpm_server_configure(0.6, 64, 256, 1000)
    for plan, wl, out in items:
        alone = plan.propagate(records=False, powers=False).psi
        assert np.linalg.norm(out - alone) <= 7.2e-6 * np.linalg.norm(alone)
        plan.close()

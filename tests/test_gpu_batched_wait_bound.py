"""The bound of device waits is the one in force at the call, also where a batch
replays a captured launch sequence: a wait that nothing completes runs out after
the bound of its own call."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["single", "pairs"])
def test_batch_after_another_bound(kernel, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as sp2

    monkeypatch.setenv("SP2_BATCHED_KERNEL", kernel)
    sp2.finalize()
    sp2.init(0)
    try:
        H = torch.diag(torch.linspace(-1, 1, 300, device="cuda")).contiguous()
        Hs, n_occ = [H, H[:200, :200].contiguous()], [150, 100]
        want, _ = sp2.density_matrix_batched(Hs, n_occ)
        want = [d.clone() for d in want]

        def seconds_to_time_out(ms):
            sp2.set_fault(f"timeout,wait_ms={ms}")
            t0 = time.perf_counter()
            with pytest.raises(sp2.SP2Error) as e:
                sp2.density_matrix_batched(Hs, n_occ)
            assert e.value.status == -7  # SP2_ERR_DEVICE_TIMEOUT
            return time.perf_counter() - t0

        assert seconds_to_time_out(1500) >= 1.5
        assert seconds_to_time_out(100) < 1.0
        assert seconds_to_time_out(1500) >= 1.5
        sp2.set_fault(None)
        got, _ = sp2.density_matrix_batched(Hs, n_occ)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    finally:
        sp2.set_fault(None)
        monkeypatch.undo()
        sp2.finalize()
        sp2.init(0)

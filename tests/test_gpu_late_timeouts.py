"""A bounded device wait that runs out in a call which returns before the end of
its work is reported by the next call, once; the library stays usable.  The wait
is on a barrier that nothing arrives on, under a 100 ms bound."""
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THETA = [(0.4, 0.9, -0.1), (-1.0, 2.0, 0.0)]
C = [0.1, -0.05, 0.2]


@pytest.fixture(params=["default", "single"])
def sp2(request, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as m

    if request.param == "single":
        monkeypatch.setenv("SP2_SQUARE_KERNEL", "single")
    m.finalize()
    m.init(0)
    yield m
    m.set_fault(None)
    monkeypatch.undo()
    m.finalize()
    m.init(0)


def _matrices(B, N):
    g = torch.Generator(device="cuda").manual_seed(N + B)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    return ((H + H.mT) / (2 * N**0.5)).contiguous()


# the resident kernel with one slot and with two, CTA pairs
SIZES = [(4, 128), (200, 96), (10, 1300)]


def _times_out_late(sp2, run):
    """run() without the fault, then with it: the call after it reports."""
    want = run()
    sp2.set_fault("timeout,wait_ms=100")
    run()
    torch.cuda.synchronize()
    sp2.set_fault(None)
    with pytest.raises(sp2.SP2Error) as e:
        run()
    assert e.value.status == -7  # SP2_ERR_DEVICE_TIMEOUT
    got = run()
    assert torch.equal(got, want)


@pytest.mark.parametrize("B,N", SIZES)
def test_forward(sp2, B, N):
    H = _matrices(B, N)
    coef = torch.tensor([[0.4, 0.9, -0.1], [-0.8, 1.5, 0.05]])
    _times_out_late(sp2, lambda: sp2.network_forward(H, coef, 1)[0])


@pytest.mark.parametrize("B,N", SIZES)
@pytest.mark.parametrize("window", [None, (-4.0, 4.0)])
def test_expansion(sp2, B, N, window):
    H = _matrices(B, N)
    _times_out_late(sp2, lambda: sp2.fermi_expansion(H, THETA, C, window)[0])


@pytest.mark.parametrize("N", [100, 700, 3000])
def test_solve_without_statistics(sp2, N):
    H = _matrices(1, N)[0].contiguous()
    _times_out_late(sp2, lambda: sp2.density_matrix(H, N // 2, sync=False)[0])


@pytest.mark.parametrize("B,N", SIZES)
def test_adjoint_after_the_forward_pass(sp2, B, N):
    H = _matrices(B, N)
    coef = torch.tensor([[0.4, 0.9, -0.1], [-0.8, 1.5, 0.05]])
    X, ck, _ = sp2.network_forward(H, coef, 1)
    want = sp2.network_backward(H, coef, 1, ck, X)
    sp2.set_fault("timeout,wait_ms=100")
    X1, ck1, _ = sp2.network_forward(H, coef, 1)
    with pytest.raises(sp2.SP2Error) as e:  # its checkpoints are not valid
        sp2.network_backward(H, coef, 1, ck1, X1)
    assert e.value.status == -7
    sp2.set_fault(None)
    got = sp2.network_backward(H, coef, 1, ck, X)
    assert torch.equal(got[1], want[1]) and torch.equal(got[0], want[0])


def test_a_reported_time_out_is_not_reported_again(sp2):
    N = 300
    H = _matrices(1, N)[0].contiguous()
    want, _ = sp2.density_matrix(H, N // 2)
    sp2.set_fault("timeout,wait_ms=100")
    with pytest.raises(sp2.SP2Error) as e:
        sp2.density_matrix(H, N // 2)
    assert e.value.status == -7
    sp2.set_fault(None)
    assert torch.equal(sp2.density_matrix(H, N // 2)[0], want)

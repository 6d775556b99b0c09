"""The adjoint's workspace: in proportion to what the header states, and the CTA
pairs' path where the resident one's does not fit."""
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def sp2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as m

    m.finalize()  # no workspace
    m.init(0)
    yield m
    m.set_fault(None)
    m.finalize()
    m.init(0)


def _inputs(B, N, L):
    g = torch.Generator(device="cuda").manual_seed(N + B)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous()
    G = torch.randn(B, N, N, generator=g, device="cuda") / N
    coef = torch.rand(L, 3, generator=torch.Generator().manual_seed(L)) * 0.3 + torch.tensor([0.1, 0.3, -0.1])
    return H, (G + G.mT).contiguous(), coef


def _single(fn):
    import paper_2101_06385_gb300 as sp2

    os.environ["SP2_SQUARE_KERNEL"] = "single"
    sp2.finalize()
    sp2.init(0)
    try:
        return fn(sp2)
    finally:
        del os.environ["SP2_SQUARE_KERNEL"]
        sp2.finalize()
        sp2.init(0)


def _equal(got, want):
    assert torch.equal(got[1], want[1])
    # FP64 sums of the same FP32 parts in another order
    assert torch.allclose(got[0], want[0], rtol=1e-12, atol=1e-12 * float(want[0].abs().max()))


# many tiny matrices in one long segment: whole tiles of iterates would be 69 GB
def test_tiny_matrices_long_segment(sp2):
    B, N, L, ce = 4096, 1, 256, 256
    H, G, coef = _inputs(B, N, L)
    X, ck, _ = sp2.network_forward(H, coef, ce)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    got = sp2.network_backward(H, coef, ce, ck, G)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 7 << 30
    _equal(got, _single(lambda m: m.network_backward(H, coef, ce, ck, G)))


def test_refused_planes_go_to_the_pairs(sp2):
    B, N, L, ce = 8, 512, 20, 1  # planes of 22 iterates: 92 MB each; 12.6 MB on the pairs
    H, G, coef = _inputs(B, N, L)
    X, ck, _ = sp2.network_forward(H, coef, ce)
    want = sp2.network_backward(H, coef, ce, ck, G)
    sp2.finalize()
    sp2.init(0)
    sp2.set_fault("alloc_limit=40")
    _equal(sp2.network_backward(H, coef, ce, ck, G), want)
    sp2.set_fault(None)
    _equal(sp2.network_backward(H, coef, ce, ck, G), want)


def test_injected_allocation_failure_is_reported(sp2):
    B, N, L, ce = 2, 64, 3, 1
    H, G, coef = _inputs(B, N, L)
    X, ck, _ = sp2.network_forward(H, coef, ce)
    sp2.set_fault("alloc_fail")
    with pytest.raises(sp2.SP2Error) as e:
        sp2.network_backward(H, coef, ce, ck, G)
    assert e.value.status == -6  # SP2_ERR_OOM
    _equal(sp2.network_backward(H, coef, ce, ck, G), _single(lambda m: m.network_backward(H, coef, ce, ck, G)))

"""Where a cooperative launch is refused (a process or stream with too few SMs for
the kernels whose CTAs wait on one another) every call runs with a launch a layer
instead, with the same results.  The refusal is injected on the host."""
import pytest

import sp2_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as m

    m.init(0)
    yield m
    m.set_fault(None)


def _both(sp2, run):
    sp2.set_fault(None)
    want = run()
    sp2.set_fault("no_cooperative")
    try:
        return run(), want
    finally:
        sp2.set_fault(None)


# the resident kernel and lists of layers on the CTA pairs
@pytest.mark.parametrize("N", [100, 1021, 3100])
@pytest.mark.parametrize("mode", ["split", "fp16", "fp32", "accelerated"])
def test_single_solve(sp2, N, mode):
    n_occ = N // 3
    h = si.gapped_hamiltonian(N, n_occ, (-1.0, -0.1), (0.1, 1.0), seed=N, device="cuda" if N > 1000 else "cpu")
    H = torch.from_numpy(h.h32()).cuda()

    def solve():
        if mode == "accelerated":
            return sp2.density_matrix_accelerated(H, n_occ, -0.1, 0.1, precision="split")
        return sp2.density_matrix(H, n_occ, precision=mode)

    (D, st), (D1, s1) = _both(sp2, solve)
    assert torch.equal(D, D1)
    assert st.sigmas == s1.sigmas and st.converged_by == s1.converged_by and st.status == 0
    assert all(t > 0 for t in st.layer_ms[: st.iterations])


def test_batch(sp2):
    sizes = [700, 64, 300, 129] * 3
    Hs = [torch.from_numpy(si.gapped_hamiltonian(N, N // 2, (-1.0, -0.1), (0.1, 1.0), seed=N).h32()).cuda() for N in sizes]
    (Ds, st), (D1, s1) = _both(sp2, lambda: sp2.density_matrix_batched(Hs, [N // 2 for N in sizes]))
    assert all(torch.equal(a, b) for a, b in zip(Ds, D1))
    assert [s.sigmas for s in st] == [s.sigmas for s in s1]


@pytest.mark.parametrize("B,N", [(8, 128), (3, 257), (12, 1300)])
def test_network_and_expansion(sp2, B, N):
    g = torch.Generator(device="cuda").manual_seed(N)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous()
    G = torch.randn(B, N, N, generator=g, device="cuda") / N
    G = (G + G.mT).contiguous()
    coef = torch.tensor([[0.4, 0.9, -0.1], [-0.8, 1.5, 0.05], [0.7, 0.3, 0.0], [-0.5, 1.2, 0.1], [0.9, 0.1, 0.0]])

    def run():
        X, ck, bounds = sp2.network_forward(H, coef, 2)
        dcoef, G0 = sp2.network_backward(H, coef, 2, ck, G)
        D, _ = sp2.fermi_expansion(H, [(0.4, 0.9, -0.1), (-1.0, 2.0, 0.0), (0.8, 0.1, 0.0)], [0.1, -0.05, 0.2, 0.3])
        return X, ck, bounds, G0, dcoef, D

    got, want = _both(sp2, run)
    for a, b in zip(got[:4], want[:4]):
        assert torch.equal(a, b)
    # FP64 sums of the same FP32 parts in another order; one rounding to FP32
    assert torch.allclose(got[4], want[4], rtol=1e-12, atol=1e-12 * float(want[4].abs().max()))
    assert float((got[5] - want[5]).abs().max()) <= 2**-23 * float(want[5].abs().max())

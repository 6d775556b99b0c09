"""Lists of layers on CTA pairs (one launch per list, tiles of a layer started
when their matrix has finished the layer before) against the single-CTA kernel,
one launch per layer: the same bits, for sizes that take this path."""
import time

import pytest

import sp2_inputs as si
from test_gpu_resident import _with_env, sp2  # noqa: F401  (the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve_input(N):
    n_occ = N // 3
    h = si.gapped_hamiltonian(N, n_occ, (-1.0, -0.1), (0.1, 1.0), seed=500 + N, device="cuda")
    return torch.from_numpy(h.h32()).cuda(), n_occ


# the smallest size of the path (odd rows), a last column of one, wide units
# (a row's odd last tile without a partner)
@pytest.mark.parametrize("N,wide", [(2945, "0"), (3073, "0"), (2945, "1"), (3400, "1")])
@pytest.mark.parametrize("mode", ["split", "fp16", "accelerated"])
def test_solve_same_bits(sp2, N, wide, mode):  # noqa: F811
    H, n_occ = _solve_input(N)

    def solve(m):
        if mode == "accelerated":
            return m.density_matrix_accelerated(H, n_occ, -0.1, 0.1, precision="split")
        return m.density_matrix(H, n_occ, precision=mode)

    D, st = _with_env("SP2_WIDE", wide, solve)
    D1, s1 = _with_env("SP2_SQUARE_KERNEL", "single", solve)
    assert torch.equal(D, D1)
    assert st.sigmas == s1.sigmas and st.converged_by == s1.converged_by and st.energy == pytest.approx(s1.energy)
    ran = st.iterations + (0 if mode == "accelerated" else 2)
    assert all(t > 0 for t in st.layer_ms[:ran]) and not any(st.layer_ms[ran:])


@pytest.mark.parametrize("max_iter", [1, 2, 3])
def test_last_layers(sp2, max_iter):  # noqa: F811
    H, n_occ = _solve_input(2945)
    run = lambda m: m.density_matrix(H, n_occ, max_iter=max_iter)  # noqa: E731
    (D, st), (D1, s1) = run(sp2), _with_env("SP2_SQUARE_KERNEL", "single", run)
    assert torch.equal(D, D1) and (st.status, st.iterations) == (s1.status, s1.iterations)


# several uneven groups of matrices, one group, a matrix larger than a group;
# segments of one layer, of several, and as long as the network
@pytest.mark.parametrize("B,N,L,ce", [(20, 1100, 5, 2), (13, 1000, 4, 1), (7, 1793, 6, 4), (2, 3000, 3, 3)])
@pytest.mark.parametrize("precision", ["split", "fp16"])
def test_network_same_bits(sp2, B, N, L, ce, precision):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(N + B)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous() + torch.diag(torch.linspace(-1, 1, N, device="cuda"))
    G = torch.randn(B, N, N, generator=g, device="cuda") / N
    G = (G + G.mT).contiguous()
    coef = torch.rand(L, 3, generator=torch.Generator().manual_seed(L)) - torch.tensor([0.5, 0.0, 0.5])

    def run(m):
        m.set_precision(precision)
        X, ck, bounds = m.network_forward(H, coef, ce)
        dcoef, G0 = m.network_backward(H, coef, ce, ck, G)
        m.set_precision("split")
        return X, ck, bounds, G0, dcoef

    got, want = run(sp2), _with_env("SP2_SQUARE_KERNEL", "single", run)
    for a, b in zip(got[:4], want[:4]):
        assert torch.equal(a, b)
    # FP64 sums of the same FP32 parts in another order
    assert torch.allclose(got[4], want[4], rtol=1e-12, atol=1e-12 * float(want[4].abs().max()))


# the expansion has no single-CTA path: against its layers in FP64 on the GPU's
# matrix product, each split layer adding at most 2^-20 of the operands' norm
@pytest.mark.parametrize("B,N", [(14, 1300), (7, 1793), (2, 3000)])
def test_expansion(sp2, B, N):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(N + B)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous() + torch.diag(torch.linspace(-1, 1, N, device="cuda"))
    theta = [(0.4, 0.9, -0.1), (-1.0, 2.0, 0.0), (1.0, 0.0, 0.05), (-0.7, 1.5, 0.1)]
    c = [0.1, -0.05, 0.2, 0.3, 0.5]
    D, _ = sp2.fermi_expansion(H, theta, c, (-4.0, 4.0))
    one = torch.eye(N, device="cuda", dtype=torch.float64)
    for b in {0, B // 2, B - 1}:
        X = (H[b].double() + 4.0 * one) / 8.0
        R = c[0] * X
        for (p, q, r), w in zip(theta, c[1:]):
            X = p * X @ X + q * X + r * one
            R = R + w * X
        assert float((D[b].double() - (one - R)).abs().max()) <= len(theta) * 2**-20


def test_wait_runs_out(sp2):  # noqa: F811
    H, n_occ = _solve_input(2945)
    try:
        sp2.set_fault("timeout,wait_ms=100")
        t0 = time.perf_counter()
        with pytest.raises(sp2.SP2Error) as e:
            sp2.density_matrix(H, n_occ)
        assert e.value.status == -7 and time.perf_counter() - t0 < 30.0
    finally:
        sp2.set_fault(None)
    D, st = sp2.density_matrix(H, n_occ)
    assert st.status == 0 and abs(float(D.diagonal().double().sum()) - n_occ) < 1e-2

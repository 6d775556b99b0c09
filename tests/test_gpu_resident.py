"""The resident solve (all layers of a batch in one launch on 128 x 128 tiles)
against the launch-per-layer kernels it takes over from: the same bits, at the
edges of its tiles and of its range."""
import os

import numpy as np
import pytest

import oracle as o
import sp2_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _with_env(name, value, fn):
    import paper_2101_06385_gb300 as sp2

    os.environ[name] = value
    sp2.finalize()
    sp2.init(0)
    try:
        return fn(sp2)
    finally:
        del os.environ[name]
        sp2.finalize()
        sp2.init(0)


@pytest.fixture(scope="module")
def sp2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as m

    m.init(0)
    return m


# one tile, its edge, a lone last row and column of tiles, the lower tile of a
# diagonal super tile, odd rows, more tiles than CTAs, the largest size
@pytest.mark.parametrize("N", [1, 31, 128, 129, 257, 385, 1021, 2053, 2816])
@pytest.mark.parametrize("mode", ["split", "fp16", "accelerated"])
def test_single_solve_same_bits(sp2, N, mode):
    n_occ = max(1, N // 3)
    h = si.gapped_hamiltonian(N, n_occ, (-1.0, -0.1), (0.1, 1.0), seed=300 + N, device="cuda" if N > 1000 else "cpu")
    H = torch.from_numpy(h.h32()).cuda()

    def solve(m):
        if mode == "accelerated":
            return m.density_matrix_accelerated(H, n_occ, -0.1, 0.1, precision="split")
        return m.density_matrix(H, n_occ, precision=mode)

    D, st = solve(sp2)
    D1, s1 = _with_env("SP2_SQUARE_KERNEL", "single", solve)
    assert torch.equal(D, D1)
    assert st.sigmas == s1.sigmas and st.converged_by == s1.converged_by
    # times of the layers it ran, none after them
    ran = st.iterations + (0 if mode == "accelerated" else 2)
    assert all(t > 0 for t in st.layer_ms[:ran]) and not any(st.layer_ms[ran:])


# FP32 on the CUDA cores: tiles of 32 (one a CTA, several) and of 64, their
# edges, rows that are no multiple of four
@pytest.mark.parametrize("N", [1, 2, 32, 33, 129, 511, 514, 900, 1021, 1920])
@pytest.mark.parametrize("accelerated", [False, True])
def test_fp32_solve_same_bits(sp2, N, accelerated):
    n_occ = max(1, N // 3)
    h = si.gapped_hamiltonian(N, n_occ, (-1.0, -0.1), (0.1, 1.0), seed=500 + N, device="cuda" if N > 1000 else "cpu")
    H = torch.from_numpy(h.h32()).cuda()

    def solve(m):
        if accelerated:
            return m.density_matrix_accelerated(H, n_occ, -0.1, 0.1, precision="fp32")
        return m.density_matrix(H, n_occ, precision="fp32")

    D, st = solve(sp2)
    D1, s1 = _with_env("SP2_SQUARE_KERNEL", "single", solve)
    assert torch.equal(D, D1)
    assert st.sigmas == s1.sigmas and st.converged_by == s1.converged_by and st.status == 0


def test_layer_limits(sp2):
    """One layer and an early stop: the launch that writes D comes first, or second."""
    h = si.gapped_hamiltonian(200, 80, (-1.0, -0.1), (0.1, 1.0), seed=520)
    H = torch.from_numpy(h.h32()).cuda()
    for prec in ("split", "fp32"):
        for solve in (
            lambda m: m.density_matrix(H, 80, max_iter=1, precision=prec),
            lambda m: m.density_matrix_accelerated(H, 80, -0.1, 0.1, max_iter=1, precision=prec),
            lambda m: m.density_matrix_accelerated(H, 80, -0.1, 0.1, max_iter=2, precision=prec),
        ):
            try:
                got = solve(sp2)
            except sp2.SP2Error as e:  # one layer leaves Tr D far from N_occ
                got = e.status
            try:
                want = _with_env("SP2_SQUARE_KERNEL", "single", solve)
            except sp2.SP2Error as e:
                want = e.status
            if isinstance(want, int):
                assert got == want
            else:
                assert torch.equal(got[0], want[0]) and got[1].status == want[1].status


# an instance on both slots of every CTA among small ones, and more instances
# than slots (each slot works through a list)
@pytest.mark.parametrize("sizes", [[2500, 64, 700, 1, 300], [1000, 96] * 20 + [130] * 300 + [7, 513]])
def test_batch_same_bits(sp2, sizes):
    kinds = {N: si.gapped_hamiltonian(N, N // 2, (-1.0, -0.05), (0.05, 1.0), seed=400 + N) for N in set(sizes)}
    Hs = [torch.from_numpy(kinds[N].h32()).cuda() for N in sizes]
    n_occ = [N // 2 for N in sizes]
    Ds, st = sp2.density_matrix_batched(Hs, n_occ)
    Dp, sp = _with_env("SP2_BATCHED_KERNEL", "pairs", lambda m: m.density_matrix_batched(Hs, n_occ))
    for a, b in zip(Ds, Dp):
        assert torch.equal(a, b)
    assert [s.sigmas for s in st] == [s.sigmas for s in sp]
    m = o.error_metrics(Ds[0].cpu().numpy().astype(np.float64), o.density_matrix_closed_form(kinds[sizes[0]].Q, n_occ[0]),
                        n_occ[0])
    assert m["max_abs"] <= 5e-5 and m["trace_err"] <= 1e-4, m


def test_input_that_is_not_symmetric_stops_alike(sp2):
    """Symmetry is assumed, not checked: an iterate that leaves the range of the
    layer's fixed-point sums stops the solve as it does on the other kernels."""
    N = 300
    H = torch.zeros(N, N, device="cuda")
    H += torch.diag(torch.linspace(-1, 1, N, device="cuda"))
    H[: N // 2, N // 2:] = 5.0  # the rows' bounds hold for H, not for its upper triangle mirrored
    D, st = sp2.density_matrix(H, N // 2)
    D1, s1 = _with_env("SP2_SQUARE_KERNEL", "single", lambda m: m.density_matrix(H, N // 2))
    assert st.status == s1.status and st.converged_by == s1.converged_by


# one matrix a CTA, gangs, more matrices than slots; segments of one layer, of
# several, longer than the network; sizes off every boundary
@pytest.mark.parametrize("B,N,L,ce", [(8, 128, 7, 3), (1, 1, 3, 1), (3, 257, 5, 2), (5, 100, 6, 1), (2, 1000, 4, 4),
                                      (400, 40, 3, 2), (1, 2053, 3, 2), (20, 700, 3, 2), (100, 40, 3, 2)])
@pytest.mark.parametrize("precision", ["split", "fp16"])
def test_network_same_bits(sp2, B, N, L, ce, precision):
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


@pytest.mark.parametrize("B,N", [(1, 1), (3, 130), (2, 1000), (200, 64), (1, 2053)])
@pytest.mark.parametrize("window", [None, (-4.0, 4.0)])
def test_expansion_same_values(sp2, B, N, window):
    g = torch.Generator(device="cuda").manual_seed(N + B)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous() + torch.diag(torch.linspace(-1, 1, N, device="cuda"))
    theta = [(0.4, 0.9, -0.1), (-1.0, 2.0, 0.0), (1.0, 0.0, 0.05), (-0.7, 1.5, 0.1)]
    c = [0.1, -0.05, 0.2, 0.3, 0.5]
    D, bounds = sp2.fermi_expansion(H, theta, c, window)
    D1, b1 = _with_env("SP2_SQUARE_KERNEL", "single", lambda m: m.fermi_expansion(H, theta, c, window))
    # the diagonal's FP64 row norms add in another order: one rounding to FP32 at most
    assert torch.equal(bounds, b1)
    assert float((D - D1).abs().max()) <= 2**-23 * float(D1.abs().max())

"""Iterates beyond the FP16 range of the operand planes (|Y| >= 2^(16 - s)): the
resident kernels leave infinities and NaN where the launch-per-layer kernels do,
and a solve that runs into them ends alike."""
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2101_06385_gb300 as m

    m.init(0)
    return m


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


@pytest.mark.parametrize("precision", ["split", "fp16"])
@pytest.mark.parametrize("N", [2, 40, 300])
def test_network(sp2, N, precision):
    B, L = 4, 6
    g = torch.Generator(device="cuda").manual_seed(N)
    H = torch.randn(B, N, N, generator=g, device="cuda")
    H = ((H + H.mT) / (2 * N**0.5)).contiguous() + torch.diag(torch.linspace(1, 3, N, device="cuda"))
    coef = torch.tensor([[1.0, 2.0, 1.0]] * L)  # squares grow past every range

    def run(m):
        m.set_precision(precision)
        X, ck, _ = m.network_forward(H, coef, 1)
        m.set_precision("split")
        return X.clone(), ck.clone()

    got, want = run(sp2), _single(run)
    assert not want[0].isfinite().all() and want[1][1].isfinite().all()
    for a, b in zip(got, want):
        assert torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(0.0), b.nan_to_num(0.0))


def test_solve_of_two(sp2):
    for lo in (2.0, 5.0):
        H = torch.tensor([[lo, 0.3], [0.3, lo + 1.0]], device="cuda")
        run = lambda m: m.density_matrix(H, 1)
        (D, st), (D1, s1) = run(sp2), _single(run)
        assert (st.status, st.converged_by, st.sigmas) == (s1.status, s1.converged_by, s1.sigmas)
        assert torch.equal(D.isnan(), D1.isnan()) and torch.equal(D.nan_to_num(0.0), D1.nan_to_num(0.0))

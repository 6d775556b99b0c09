"""Spectra that lie on one side of zero.  The input layer then starts with a
shift outside [0, 1], and the iterate Y = S - alpha I of the first layers is
larger than 1: the resident solves' sums leave their fixed-point range and have
to be the same all the same as the launch-per-layer kernels' FP64 sums."""
import os

import numpy as np
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


def _launch_per_layer(fn):
    import paper_2101_06385_gb300 as sp2

    names = ("SP2_SQUARE_KERNEL", "SP2_BATCHED_KERNEL")
    for n in names:
        os.environ[n] = "single"
    sp2.finalize()
    sp2.init(0)
    try:
        return fn(sp2)
    finally:
        for n in names:
            del os.environ[n]
        sp2.finalize()
        sp2.init(0)


def _tridiagonal(N, n_occ, lo, seed):
    """Eigenvalues near [lo, lo + 2] with a gap of 0.4 (tight Gershgorin bounds), FP64 projector."""
    rng = np.random.default_rng(seed)
    mid = lo + 2.0 * n_occ / N
    d = rng.permutation(np.concatenate([rng.uniform(lo, mid - 0.2, n_occ), rng.uniform(mid + 0.2, lo + 2, N - n_occ)]))
    h = np.diag(d)
    i = np.arange(N - 1)
    h[i, i + 1] = h[i + 1, i] = 0.02
    h = h.astype(np.float32)
    _, v = np.linalg.eigh(h.astype(np.float64))
    return h, v[:, :n_occ] @ v[:, :n_occ].T, mid


def _outcome(fn):
    from paper_2101_06385_gb300 import SP2Error

    try:
        return fn()
    except SP2Error as e:
        return e.status


def _same(got, want, exact, tol):
    """The same end; D as close to the projector where the reference kernels are."""
    if isinstance(want, int):
        assert got == want
        return None
    assert not isinstance(got, int), got
    (D, st), (D1, s1) = got, want
    assert st.status == s1.status and st.converged_by == s1.converged_by and st.sigmas == s1.sigmas
    assert np.isfinite(st.trace) == np.isfinite(s1.trace)
    err = float(np.abs(D1.cpu().numpy() - exact).max())
    if err <= tol:
        assert float(np.abs(D.cpu().numpy() - exact).max()) <= tol
        assert abs(st.trace - s1.trace) <= 1e-9 * max(1.0, abs(s1.trace))
    return err <= tol


# one tile, gangs of one slot, gangs of two
@pytest.mark.parametrize("N", [64, 200, 1100, 2100])
@pytest.mark.parametrize("mode", ["split", "fp16", "accelerated"])
def test_single_solve(sp2, N, mode):
    right = 0
    for lo in (0.2, 1.0, -3.0, 4.0):
        for frac in (0.2, 0.5, 0.8) if N < 1000 else (0.5,):
            n_occ = int(N * frac)
            h, exact, mid = _tridiagonal(N, n_occ, lo, N + n_occ)
            H = torch.from_numpy(h).cuda()

            def solve(m):
                if mode == "accelerated":
                    return m.density_matrix_accelerated(H, n_occ, mid - 0.15, mid + 0.15, precision="split")
                return m.density_matrix(H, n_occ, precision=mode)

            got, want = _outcome(lambda: solve(sp2)), _outcome(lambda: _launch_per_layer(solve))
            right += bool(_same(got, want, exact, 2e-3 if mode == "fp16" else 5e-5))
    assert right >= 2  # the reference kernels solve some of them


def test_batch(sp2):
    cases = [_tridiagonal(N, N // 2, lo, N) for N in (64, 130, 300, 777) for lo in (-1.0, 0.2, 1.0, -2.8)]
    Hs = [torch.from_numpy(c[0]).cuda() for c in cases]
    n_occ = [len(c[0]) // 2 for c in cases]
    run = lambda m: m.density_matrix_batched(Hs, n_occ)
    got, want = run(sp2), _launch_per_layer(run)
    right = sum(bool(_same((got[0][i], got[1][i]), (want[0][i], want[1][i]), cases[i][1], 5e-5)) for i in range(len(cases)))
    assert right >= 8


def test_wild_input_stops_alike(sp2):
    """An H that is not symmetric leaves the range by many orders of magnitude."""
    N = 300
    for amp in (5.0, 1e4):
        H = torch.diag(torch.linspace(-1, 1, N, device="cuda")).contiguous()
        H[: N // 2, N // 2:] = amp
        for prec in ("split", "fp16"):
            run = lambda m: m.density_matrix(H, N // 2, precision=prec)
            (_, st), (_, s1) = run(sp2), _launch_per_layer(run)
            assert (st.status, st.converged_by, st.iterations) == (s1.status, s1.converged_by, s1.iterations)
            # (the kernels read different triangles of it: no value to compare)
            assert np.isnan(st.trace) == np.isnan(s1.trace)
            acc = lambda m: m.density_matrix_accelerated(H, N // 2, -0.1, 0.1, precision=prec)
            assert _outcome(lambda: acc(sp2)) == _outcome(lambda: _launch_per_layer(acc))


# FP32: tiles of 32, one a CTA and several, and of 64
@pytest.mark.parametrize("N", [64, 200, 700, 1100])
@pytest.mark.parametrize("accelerated", [False, True])
def test_fp32_solve(sp2, N, accelerated):
    right = 0
    for lo in (0.2, 1.0, -3.0, 4.0):
        for frac in (0.2, 0.5, 0.8) if N < 1000 else (0.5,):
            n_occ = int(N * frac)
            h, exact, mid = _tridiagonal(N, n_occ, lo, N + n_occ)
            H = torch.from_numpy(h).cuda()

            def solve(m):
                if accelerated:
                    return m.density_matrix_accelerated(H, n_occ, mid - 0.15, mid + 0.15, precision="fp32")
                return m.density_matrix(H, n_occ, precision="fp32")

            got, want = _outcome(lambda: solve(sp2)), _outcome(lambda: _launch_per_layer(solve))
            right += bool(_same(got, want, exact, 5e-5))
    assert right >= 1


@pytest.mark.parametrize("N", [1, 24, 308, 1100])
@pytest.mark.parametrize("precision", ["split", "fp16", "fp32"])
def test_no_state_or_every_state_occupied(sp2, N, precision):
    """S goes to 0 or I, the sums of Y below the fixed-point units: as many layers all the same."""
    import paper_2101_06385_gb300 as m

    h = _tridiagonal(N, N // 2, -1.0, N)[0] if N > 1 else np.array([[0.3]], dtype=np.float32)
    H = torch.from_numpy(h).cuda()
    for shift in (True, False):
        for n_occ in (0, N):

            def solve(single):
                if single:
                    os.environ["SP2_SQUARE_KERNEL"] = "single"
                try:
                    m.finalize()
                    m.init(0, shift_identity=shift)
                    return m.density_matrix(H, n_occ, precision=precision)
                finally:
                    os.environ.pop("SP2_SQUARE_KERNEL", None)

            (D, st), (D1, s1) = solve(False), solve(True)
            assert (st.status, st.converged_by, st.iterations) == (s1.status, s1.converged_by, s1.iterations)
            assert float((D - D1).abs().max()) <= 1e-6
            assert abs(st.trace - n_occ) <= 1e-6 * max(1, n_occ)
    m.finalize()
    m.init(0)

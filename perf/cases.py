"""Performance cases: the work that a user of this library has it do.

A case is a dict of plain values.  Four kinds, each through the public Python
entry points:

* ``solve``    one Hamiltonian to its density matrix (``density_matrix``, or
               ``density_matrix_accelerated`` with HOMO / LUMO estimates),
* ``batched``  many Hamiltonians of uneven size (``density_matrix_batched``),
* ``fermi``    finite-temperature expansion with readout (``fermi_expansion``),
* ``network``  one training step of the Eq. 16 network: forward, loss
               gradient, adjoint.

The Hamiltonians are dense with a known gapped spectrum, H = Q diag(eps) Q^T.
Q is a product of random orthogonal circulants and random signs, applied by
FFTs in float64, so that an N = 16384 matrix takes a fraction of a second and
the exact density matrix is known without a diagonalisation.
"""
import math

import numpy as np
import torch

import paper_2101_06385_gb300 as sp2

# Fitted coefficients of an 11-layer expansion of the Fermi function at
# beta = 40 on the unit energy window (six digits): layers, then the readout.
_FERMI_THETA = [
    (1.202454, 0.194052, 0.117023), (-0.841352, 2.012818, -0.040880), (0.987099, -0.074561, -0.106392),
    (-0.977635, 2.024899, -0.041652), (1.038469, -0.072809, -0.002496), (-1.073283, 2.010114, 0.004079),
    (1.033958, 0.007552, -0.023394), (-1.056579, 1.993961, 0.003431), (1.012304, 0.025738, 0.163464),
    (-1.067926, 1.909250, -0.044128), (0.757576, -0.112978, -0.193037),
]
_FERMI_C = [-0.009499, 0.004302, 0.180640, -0.083650, -0.074227, 0.042851, 0.025256, 0.009030, 0.140380, 0.662557,
            -0.126886, 0.797695]
_KT = 0.05  # temperature of the network's target, in units of H


def listed():
    return [
        # The smallest everyday call: one N = 128 matrix (the FP64-checked
        # configuration, and every step of a small molecular-dynamics run).
        dict(name="solve_n128", kind="solve", n=128, n_occ=64, half_gap=0.1, top=1.0, precision="split",
             accelerated=False),
        # An ordinary molecule; rows that are no multiple of the tile or of 64.
        dict(name="solve_n1000", kind="solve", n=1000, n_occ=500, half_gap=0.05, top=1.0, precision="split",
             accelerated=False),
        # The mid-size configuration.
        dict(name="solve_n4096", kind="solve", n=4096, n_occ=2048, half_gap=0.05, top=1.0, precision="split",
             accelerated=False),
        # The largest configuration, the benchmark's headline.
        dict(name="solve_n16384", kind="solve", n=16384, n_occ=8192, half_gap=0.025, top=2.0, precision="split",
             accelerated=False),
        # Accelerated layers, with band-edge estimates from an earlier step of
        # a dynamics run; an odd size, so no row is 16-byte aligned.
        dict(name="accel_n2053", kind="solve", n=2053, n_occ=1026, half_gap=0.05, top=1.0, precision="split",
             accelerated=True),
        # Plain FP16 products: the fast option where 1e-3 is enough.
        dict(name="fp16_n2048", kind="solve", n=2048, n_occ=1024, half_gap=0.05, top=1.0, precision="fp16",
             accelerated=False),
        # FP32 on the CUDA cores: the comparator option.
        dict(name="fp32_n512", kind="solve", n=512, n_occ=200, half_gap=0.05, top=1.0, precision="fp32",
             accelerated=False),
        # The batched workload: 512 matrices, N in {64, 96, ..., 1024}.
        dict(name="batched_512", kind="batched", batch=512, n_min=64, n_max=1024, step=32, size_seed=1),
        # A small batch of small molecules, any size.
        dict(name="batched_16", kind="batched", batch=16, n_min=33, n_max=400, step=1, size_seed=2),
        # Finite-temperature expansion on the batch of the benchmark.
        dict(name="fermi_b64_n2048", kind="fermi", batch=64, n=2048),
        # The training workload of the benchmark.
        dict(name="network_b64_n2048", kind="network", batch=64, n=2048, layers=20, ckpt_every=5, autograd=False),
        # A small training step through torch autograd: 16 layers learnt on 8
        # matrices of N = 128.
        dict(name="network_b8_n128", kind="network", batch=8, n=128, layers=16, ckpt_every=4, autograd=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """A case of the ranges above: single solves from N = 64 to 16384, batches
    of 4 to 512, expansions and networks of 1 to 64 matrices up to 2048."""
    kind = rng.choice(["solve"] * 5 + ["batched"] * 2 + ["fermi"] + ["network"] * 2)
    if kind == "solve":
        option = rng.choice(["split"] * 5 + ["accelerated", "accelerated", "fp16", "fp32"])
        n = _log_int(rng, 64, 1024 if option == "fp32" else 16384)
        return dict(kind="solve", n=n, n_occ=max(1, int(n * rng.uniform(0.2, 0.8))),
                    half_gap=round(rng.uniform(0.025, 0.15), 4), top=round(rng.uniform(0.8, 2.0), 3),
                    precision="split" if option == "accelerated" else option, accelerated=option == "accelerated")
    if kind == "batched":
        n_min, n_max = sorted((_log_int(rng, 32, 1024), _log_int(rng, 32, 1024)))
        return dict(kind="batched", batch=_log_int(rng, 4, 512), n_min=n_min, n_max=n_max,
                    step=rng.choice([1, 32]), size_seed=rng.randrange(1 << 20))
    batch, n = _log_int(rng, 1, 64), _log_int(rng, 64, 2048)
    if kind == "fermi":
        return dict(kind="fermi", batch=batch, n=n)
    return dict(kind="network", batch=batch, n=n, layers=rng.randrange(8, 21), ckpt_every=rng.randrange(1, 6),
                autograd=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
class _Rotation:
    """Random orthogonal Q = C_1 S_1 C_2 S_2 C_3 on the last-but-one dimension
    (C: orthogonal circulant with random phases, S: random signs), one per
    matrix of a batch."""

    def __init__(self, n, batch, gen):
        h = n // 2 + 1
        phase = torch.rand((3, batch, h, 1), generator=gen, device="cuda", dtype=torch.float64) * (2 * math.pi)
        # the zero and (n even) the Nyquist frequency are real
        ends = [0] + ([h - 1] if n % 2 == 0 else [])
        phase[:, :, ends] = (phase[:, :, ends] < math.pi).double() * math.pi
        self.n = n
        self.phase = torch.polar(torch.ones_like(phase), phase)
        self.sign = torch.randint(0, 2, (2, batch, n, 1), generator=gen, device="cuda").double() * 2 - 1

    def _circulant(self, x, phase):
        return torch.fft.irfft(torch.fft.rfft(x, dim=-2).mul_(phase), n=self.n, dim=-2)

    def q(self, x):
        for k in (2, 1, 0):
            x = self._circulant(x, self.phase[k])
            if k:
                x *= self.sign[k - 1]
        return x

    def qt(self, x):
        for k in (0, 1, 2):
            if k:
                x = x * self.sign[k - 1]
            x = self._circulant(x, self.phase[k].conj())
        return x

    def matrix(self, values):
        """Q diag(values) Q^T for values [batch, n], in float64."""
        eye = torch.eye(self.n, dtype=torch.float64, device="cuda").expand(values.shape[0], -1, -1)
        m = self.q(self.qt(eye).mul_(values[:, :, None]))
        return (m + m.mT).mul_(0.5)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _spectrum(n, n_occ, half_gap, top, gen):
    """Ascending eigenvalues: n_occ uniform in [-top, -half_gap], the others in
    [half_gap, top]; half_gap is a number or one per matrix of a batch [B, 1]."""
    half_gap = torch.as_tensor(half_gap, dtype=torch.float64, device="cuda").reshape(-1, 1)
    u = torch.rand((half_gap.shape[0], n), generator=gen, device="cuda", dtype=torch.float64)
    eps = half_gap + (top - half_gap) * u
    eps[:, :n_occ] *= -1.0
    return torch.sort(eps, dim=1).values


def _problems(case, seed):
    """[(rotation, eigenvalues [B, n], n_occ)] of a case, one per matrix size,
    and for ``batched`` the order of its matrices."""
    gen = _generator(seed)
    if case["kind"] == "solve":
        rot = _Rotation(case["n"], 1, gen)
        return [(rot, _spectrum(case["n"], case["n_occ"], case["half_gap"], case["top"], gen), case["n_occ"])]
    if case["kind"] == "batched":
        sizes = _sizes(case)
        found = []
        for n in sorted(set(sizes)):
            count = sizes.count(n)
            gap = 0.05 + 0.25 * torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)
            rot = _Rotation(n, count, gen)
            found.append((rot, _spectrum(n, n // 2, 0.5 * gap, 1.0, gen), n // 2))
        return found
    rot = _Rotation(case["n"], case["batch"], gen)
    half_gap = torch.full((case["batch"],), 0.05)
    return [(rot, _spectrum(case["n"], case["n"] // 2, half_gap, 1.0, gen), case["n"] // 2)]


def _sizes(case):
    rng = np.random.default_rng(case["size_seed"])
    return [int(v) for v in rng.choice(np.arange(case["n_min"], case["n_max"] + 1, case["step"]), case["batch"])]


def _bounds(H):
    """Gershgorin bounds of H [B, n, n] in float64: [B, 2]."""
    H = H.double()
    d = torch.diagonal(H, dim1=1, dim2=2)
    r = H.abs().sum(2) - d.abs()
    return torch.stack([(d - r).amin(1), (d + r).amax(1)], 1)


def _branches(x, n_occ, limit):
    """Branch coefficients (a, b, c) that SP2 takes on the scaled eigenvalues x
    (a float64 array), at most ``limit`` of them; x is left at the last layer."""
    coef, last = [], [math.inf, math.inf]
    for _ in range(limit):
        s, p = float(np.sum(x)), float(np.sum(x * x))
        err = s - p
        square = abs(p - n_occ) <= abs(2 * s - p - n_occ)
        coef.append((1.0, 0.0, 0.0) if square else (-1.0, 2.0, 0.0))
        x = x * x if square else 2 * x - x * x
        if err <= 1e-11 or (len(coef) > 2 and coef[-2] != coef[-3] and err > 4.5 * last[0] ** 2):
            break
        last = [last[1], err]
    return coef


def prepare(case, seed):
    kind = case["kind"]
    sp2.init(torch.cuda.current_device())
    probs = _problems(case, seed)
    if kind == "solve":
        (rot, eps, n_occ), = probs
        H = rot.matrix(eps)[0].float().contiguous()
        state = dict(case, H=H)
        if case["accelerated"]:
            # estimates from an earlier step: inside the gap by a tenth of it
            homo, lumo = float(eps[0, n_occ - 1]), float(eps[0, n_occ])
            state.update(homo=homo + 0.1 * (lumo - homo), lumo=lumo - 0.1 * (lumo - homo))
        return state
    if kind == "batched":
        made = {rot.n: rot.matrix(eps).float() for rot, eps, _ in probs}
        used = dict.fromkeys(made, 0)
        Hs, outs, at = [], [], 0
        sizes = _sizes(case)
        # the program's own arena for the results, 64-element aligned
        flat = torch.zeros(sum((n * n + 63) // 64 * 64 for n in sizes), device="cuda")
        for n in sizes:
            Hs.append(made[n][used[n]].contiguous().clone())
            used[n] += 1
            outs.append(flat[at:at + n * n].view(n, n))
            at += (n * n + 63) // 64 * 64
        return dict(case, Hs=Hs, n_occ=[n // 2 for n in sizes], outs=outs, flat=flat)
    (rot, eps, n_occ), = probs
    H = rot.matrix(eps).float().contiguous()
    if kind == "fermi":
        return dict(case, H=H, theta=np.array(_FERMI_THETA), c=np.array(_FERMI_C))
    # the target: Fermi-Dirac matrices; coefficients start at the branches that
    # SP2 takes on the first matrix
    target = rot.matrix(torch.sigmoid(-eps / _KT)).float()
    coef = torch.tensor(_network_coef(case, H, eps), dtype=torch.float32)
    return dict(case, H=H, target=target, coef=coef)


def _network_coef(case, H, eps):
    lo, hi = _bounds(H[:1])[0].tolist()
    x = (hi - eps[0].cpu().numpy()) / (hi - lo)
    coef = _branches(x, case["n"] // 2, case["layers"])
    # layers past the convergence of a small matrix alternate
    while len(coef) < case["layers"]:
        coef.append((1.0, 0.0, 0.0) if coef[-1][0] < 0 else (-1.0, 2.0, 0.0))
    return coef


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind == "solve":
        if state["accelerated"]:
            D, _ = sp2.density_matrix_accelerated(state["H"], state["n_occ"], state["homo"], state["lumo"],
                                                  precision=state["precision"])
        else:
            D, _ = sp2.density_matrix(state["H"], state["n_occ"], precision=state["precision"])
        return D
    if kind == "batched":
        sp2.density_matrix_batched(state["Hs"], state["n_occ"], outs=state["outs"])
        return state["flat"]
    if kind == "fermi":
        return sp2.fermi_expansion(state["H"], state["theta"], state["c"])
    batch, ck = state["batch"], state["ckpt_every"]
    if state["autograd"]:
        coef = state["coef"].detach().clone().requires_grad_()
        X = sp2.SP2Network.apply(state["H"], coef, ck)
        loss = ((X - state["target"]) ** 2).sum() / batch
        loss.backward()
        return X.detach(), coef.grad
    X, kept, bounds = sp2.network_forward(state["H"], state["coef"], ck)
    G = (X - state["target"]).mul_(2.0 / batch)
    dcoef, G0 = sp2.network_backward(state["H"], state["coef"], ck, kept, G)
    return X, bounds, dcoef.float(), G0


# ------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    probs = _problems(case, seed)
    if kind == "solve":
        (rot, eps, n_occ), = probs
        occ = torch.zeros_like(eps)
        occ[:, :n_occ] = 1.0
        return rot.matrix(occ)[0]
    if kind == "batched":
        made = {}
        for rot, eps, n_occ in probs:
            occ = torch.zeros_like(eps)
            occ[:, :n_occ] = 1.0
            made[rot.n] = rot.matrix(occ)
        used = dict.fromkeys(made, 0)
        sizes = _sizes(case)
        flat = torch.zeros(sum((n * n + 63) // 64 * 64 for n in sizes), dtype=torch.float64, device="cuda")
        at = 0
        for n in sizes:
            flat[at:at + n * n] = made[n][used[n]].reshape(-1)
            used[n] += 1
            at += (n * n + 63) // 64 * 64
        return flat
    (rot, eps, n_occ), = probs
    H = rot.matrix(eps).float()
    bounds = _bounds(H)
    lo, hi = bounds[:, :1], bounds[:, 1:]
    if kind == "fermi":
        x = (eps - lo) / (hi - lo)
        f = _FERMI_C[0] * x
        for (a, b, c), r in zip(_FERMI_THETA, _FERMI_C[1:]):
            x = a * x * x + b * x + c
            f = f + r * x
        return rot.matrix(1.0 - f), bounds
    # every matrix of the training step is a function of its H, so the layers,
    # the loss gradient and the adjoint act on the eigenvalues
    coef = torch.tensor(_network_coef(case, H, eps), dtype=torch.float32).double()
    x = (hi - eps) / (hi - lo)
    kept = []
    for a, b, c in coef.tolist():
        kept.append(x)
        x = a * x * x + b * x + c
    X = rot.matrix(x)
    g = 2.0 * (x - torch.sigmoid(-eps / _KT)) / case["batch"]
    dcoef = torch.zeros_like(coef)
    for k in range(case["layers"] - 1, -1, -1):
        y = kept[k]
        dcoef[k] = torch.stack([(g * y * y).sum(), (g * y).sum(), g.sum()]).cpu()
        g = g * (2.0 * coef[k, 0].item() * y + coef[k, 1].item())
    if case["autograd"]:
        return X, dcoef
    return X, bounds, dcoef, rot.matrix(g)


# -------------------------------------------------------------------- work
def _solve_layers(n, n_occ, half_gap, top, accelerated=False):
    """Layers of a solve (with the two of the refinement), from the expected
    spectrum and the expected Gershgorin radius of a dense random H."""
    u_occ = (np.arange(n_occ) + 0.5) / n_occ
    u_virt = (np.arange(n - n_occ) + 0.5) / max(1, n - n_occ)
    eps = np.concatenate([-top + (top - half_gap) * u_occ, half_gap + (top - half_gap) * u_virt])
    rms = math.sqrt(float(np.mean(eps * eps)))
    edge = max(top, rms * math.sqrt(2.0 * n / math.pi))
    x = (edge - eps) / (2 * edge)
    if not accelerated:
        return len(_branches(x, n_occ, 100)) + 2
    l, h, count = (edge - 0.8 * half_gap) / (2 * edge), (edge + 0.8 * half_gap) / (2 * edge), 0
    while max(l, 1 - h) > 1e-9 and count < 100:
        if 1 - h <= l:
            s = 0.5 * l
            l, h = (s / (1 - s)) ** 2, ((h - s) / (1 - s)) ** 2
        else:
            t = 0.5 * (1 - h)
            l, h = 1 - ((1 - l - t) / (1 - t)) ** 2, 1 - (t / (1 - t)) ** 2
        count += 1
    return count


def work(case):
    """H in and the result out once; the products of the layers on one triangle
    (3 n^3 operations a split square, n^3 a plain one, 6 n^3 a split adjoint)."""
    kind = case["kind"]
    if kind == "solve":
        n = float(case["n"])
        layers = _solve_layers(case["n"], case["n_occ"], case["half_gap"], case["top"], case["accelerated"])
        return {"bytes": 8 * n * n, "flops": layers * (3 if case["precision"] == "split" else 1) * n ** 3}
    if kind == "batched":
        sizes = _sizes(case)
        layers = {n: _solve_layers(n, n // 2, 0.0875, 1.0) for n in set(sizes)}
        return {"bytes": sum(8.0 * n * n for n in sizes), "flops": sum(3.0 * layers[n] * n ** 3 for n in sizes)}
    per, n = float(case["batch"]), float(case["n"])
    if kind == "fermi":
        return {"bytes": 8 * per * n * n, "flops": per * 3 * n ** 3 * len(_FERMI_THETA)}
    mats = 3 if case["autograd"] else 4  # H, target and X; and the gradient at the input
    return {"bytes": 4 * mats * per * n * n, "flops": per * case["layers"] * 9 * n ** 3}

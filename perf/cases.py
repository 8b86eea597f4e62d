"""Performance cases of the density-matrix response library.

Each case is one call (or one short sequence of calls) that a user's program
makes through the Python binding on device-resident inputs: a Hamiltonian
``H = Q diag(eps) Q^T`` with a gap between its occupied and empty levels, and
symmetric perturbations, as in ``workloads.py``.  ``Q`` is here a product of
orthonormal Hartley transforms and random signs instead of the QR factor of a
Gaussian: its entries are distributed alike (variance 1/n), any size works, and
both the inputs and the exact results cost O(n^2 log n) through the FFT.

Kinds of case:

* ``response``  P and the K first-order responses of one instance
* ``orders``    the response terms of every order up to ``order``
* ``density``   P(H) with autograd: forward, and dL/dH of L = Tr[G P]
* ``batch``     many independent instances of uneven size in one call
* ``scc``       a forward run that keeps its S0 states, then the
                self-consistent response on them
"""

import math
import random

import torch

from paper_2203_09621_gb300 import dmpt

DEV = "cuda"


def listed():
    return [
        # plain FP64 perturbation theory on a small molecule (workload 1)
        dict(name="fp64_n128", kind="response", n=128, n_occ=64, k=1, gap=1.0,
             precision="fp64", h1="gauss", pad=0),
        # the same size on the tensor cores: the smallest calls, e.g. inside a
        # molecular-dynamics loop, where latency and launches count
        dict(name="fp16_n128", kind="response", n=128, n_occ=64, k=1, gap=1.0,
             precision="dual_fp16", h1="gauss", pad=0),
        # a ragged middle size with two directions
        dict(name="fp16_n1000_k2", kind="response", n=1000, n_occ=500, k=2, gap=0.2,
             precision="dual_fp16", h1="gauss", pad=0),
        # BF16 halves, three dipole directions, a fifth of the levels occupied
        dict(name="bf16_n2048_k3", kind="response", n=2048, n_occ=410, k=3, gap=0.2,
             precision="dual_bf16", h1="dipole", pad=0),
        # a water-box size with 2n/3 levels occupied: ragged, complement form
        dict(name="fp16_n5904", kind="response", n=5904, n_occ=3936, k=1, gap=0.2,
             precision="dual_fp16", h1="gauss", pad=0),
        # polarisability of a large system: three dipole directions (workload 3)
        dict(name="fp16_n8192_k3", kind="response", n=8192, n_occ=4096, k=3, gap=0.2,
             precision="dual_fp16", h1="dipole", pad=0),
        # the plain FP32 form (workload 2 compares the precisions at this size)
        dict(name="fp32_n4096", kind="response", n=4096, n_occ=2048, k=1, gap=0.2,
             precision="fp32", h1="gauss", pad=0),
        # a reference-quality FP64 run of a middle size, ragged
        dict(name="fp64_n700", kind="response", n=700, n_occ=350, k=1, gap=0.2,
             precision="fp64", h1="gauss", pad=0),
        # third-order response of a small system in two directions
        dict(name="order3_n512_k2", kind="orders", n=512, n_occ=256, k=2, order=3, gap=0.2,
             precision="dual_fp16", h1="gauss"),
        # training through P(H): forward and adjoint with checkpoints (workload 4)
        dict(name="density_n4096", kind="density", n=4096, n_occ=2048, gap=0.2,
             precision="dual_fp16", ckpt=8),
        # many molecules of uneven size at once (workload 5, half its count)
        dict(name="batch32", kind="batch", count=32, n_min=256, n_max=2048, k=1, sizes=5,
             precision="dual_fp16"),
        # self-consistent response: one forward, then response replays
        dict(name="scc_n2048_k3", kind="scc", n=2048, n_occ=1024, k=3, gap=0.2,
             precision="dual_fp16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _occ(rng, n):
    return min(n - 1, max(1, int(round(n * rng.uniform(0.1, 0.9)))))


def draw(rng):
    kind = rng.choice(["response"] * 6 + ["fp32", "fp64", "fp64", "orders", "density", "batch", "scc"])
    gap = round(rng.uniform(0.1, 0.5), 3)
    dual = rng.choice(["dual_fp16", "dual_fp16", "dual_bf16"])
    h1 = rng.choice(["gauss", "dipole"])
    pad = rng.choice([0, 0, 0, 1, 24])
    if kind == "response":
        k = rng.choice([0, 1, 1, 2, 3])
        n = _log_int(rng, 64, 7168 if k > 1 else 8192)
        return dict(kind="response", n=n, n_occ=_occ(rng, n), k=k, gap=gap, precision=dual, h1=h1, pad=pad)
    if kind == "fp32":
        k = rng.choice([1, 1, 2, 3])
        n = _log_int(rng, 64, 4096 if k == 1 else 2600)
        return dict(kind="response", n=n, n_occ=_occ(rng, n), k=k, gap=gap, precision="fp32", h1=h1, pad=pad)
    if kind == "fp64":
        k = rng.choice([0, 1, 1, 2])
        n = _log_int(rng, 32, 800)
        return dict(kind="response", n=n, n_occ=_occ(rng, n), k=k, gap=gap, precision="fp64", h1=h1, pad=pad)
    if kind == "orders":
        order = rng.choice([2, 3, 4])
        k = rng.choice([1, 2])
        n = _log_int(rng, 128, 1536)
        return dict(kind="orders", n=n, n_occ=_occ(rng, n), k=k, order=order, gap=gap, precision=dual, h1="gauss")
    if kind == "density":
        n = _log_int(rng, 128, 4096)
        return dict(kind="density", n=n, n_occ=_occ(rng, n), gap=gap, precision=dual, ckpt=rng.choice([1, 4, 8]))
    if kind == "batch":
        n_min = _log_int(rng, 64, 512)
        return dict(kind="batch", count=rng.randint(4, 32), n_min=n_min, n_max=n_min * rng.randint(2, 4), k=1,
                    sizes=rng.randrange(1 << 20), precision=dual)
    n = _log_int(rng, 256, 2048)
    return dict(kind="scc", n=n, n_occ=n // 2, k=rng.choice([1, 3]), gap=gap, precision="dual_fp16")


# ---------------------------------------------------------------------------
# Inputs


def _hartley2(a):
    """C a C with C the orthonormal discrete Hartley matrix (C = C^T = C^-1)."""
    for dim in (0, 1):
        f = torch.fft.fft(a, dim=dim, norm="ortho")
        a = f.real - f.imag
    return a


class _Basis:
    """Q = C diag(s) C diag(t) C: an orthogonal matrix applied through FFTs."""

    def __init__(self, n, g):
        self.s, self.t = ((torch.randint(0, 2, (n,), generator=g, device=DEV) * 2 - 1).to(torch.float64)
                          for _ in range(2))

    def out_of(self, a):
        """Q a Q^T."""
        a = _hartley2(a) * self.t[:, None] * self.t[None, :]
        a = _hartley2(a) * self.s[:, None] * self.s[None, :]
        return _hartley2(a)

    def into(self, a):
        """Q^T a Q."""
        a = _hartley2(a) * self.s[:, None] * self.s[None, :]
        a = _hartley2(a) * self.t[:, None] * self.t[None, :]
        return _hartley2(a)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _instance(n, n_occ, k, gap, h1, seed):
    """H, the k perturbations, and what the exact results need: the levels
    (unsorted), which of them are occupied, and the basis."""
    g = _generator(seed)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (2.0 - gap / 2) + gap / 2
    occ = torch.zeros(n, device=DEV, dtype=torch.float64)
    occ[torch.randperm(n, generator=g, device=DEV)[:n_occ]] = 1.0
    eps = torch.where(occ > 0, -u, u)
    basis = _Basis(n, g)
    H = basis.out_of(torch.diag(eps))
    H = 0.5 * (H + H.T)
    H1 = torch.empty(k, n, n, device=DEV, dtype=torch.float64)
    scale = 0.001 if h1 == "dipole" else 0.01
    xyz = torch.rand(3, n, generator=g, device=DEV, dtype=torch.float64) * 20.0
    for j in range(k):
        m = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64)
        H1[j] = (0.5 * scale) * (m + m.T)
        if h1 == "dipole":
            H1[j].diagonal().add_(xyz[j % 3])
    return H, H1, eps, occ, basis


def _padded(a, pad):
    """`a` as a view of rows with a leading dimension of n + pad."""
    if pad == 0:
        return a
    full = torch.zeros(*a.shape[:-1], a.shape[-1] + pad, device=DEV, dtype=a.dtype)
    full[..., :a.shape[-1]] = a
    return full[..., :a.shape[-1]]


def _sizes(case):
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = _log_int(r, case["n_min"], case["n_max"])
        out.append((n, round(r.uniform(0.1, 0.5), 3)))
    return out


def _loss_matrix(n, seed):
    m = torch.randn(n, n, generator=_generator(seed + 7), device=DEV, dtype=torch.float64)
    return 0.5 * (m + m.T)


def _coupling(n, seed):
    """SPD charge coupling (40 / n) / sqrt(r^2 + 1) over random coordinates."""
    x = torch.rand(n, 3, generator=_generator(seed + 11), device=DEV, dtype=torch.float64) * 20.0
    d2 = (x[:, None, :] - x[None, :, :]).square().sum(-1)
    return (40.0 / n) / torch.sqrt(d2 + 1.0)


def prepare(case, seed):
    ctx = dmpt.context(0)
    state = dict(case=case, ctx=ctx)
    kind = case["kind"]
    if kind == "batch":
        inst = [_instance(n, n // 2, case["k"], gap, "gauss", seed * 1000 + i)
                for i, (n, gap) in enumerate(_sizes(case))]
        state.update(H=[x[0] for x in inst], H1=[x[1] for x in inst],
                     n_occ=[x[0].shape[0] // 2 for x in inst])
        return state
    n = case["n"]
    if kind == "density":
        H = _instance(n, case["n_occ"], 0, case["gap"], "gauss", seed)[0]
        state.update(H=H.requires_grad_(True), G=_loss_matrix(n, seed))
        return state
    H, H1 = _instance(n, case["n_occ"], case["k"], case["gap"], case.get("h1", "dipole"), seed)[:2]
    if kind == "scc":
        opts = dmpt.options(precision=case["precision"], ckpt_every=1)
        nbytes = ctx.workspace_size(n, case["k"], opts)
        state.update(gamma=_coupling(n, seed),
                     ws=torch.empty(nbytes + 256, dtype=torch.uint8, device=DEV))
    pad = case.get("pad", 0)
    state.update(H=_padded(H, pad), H1=_padded(H1, pad))
    return state


# ---------------------------------------------------------------------------
# One pass


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind, prec = case["kind"], case["precision"]
    if kind == "response":
        P, P1, _ = ctx.sp2_response(state["H"], state["H1"] if case["k"] else None, case["n_occ"], precision=prec)
        return [P, P1]
    if kind == "orders":
        P, terms, _ = ctx.sp2_response_m(state["H"], state["H1"], case["n_occ"], case["order"], precision=prec)
        return [P, *terms]
    if kind == "density":
        P = dmpt.density(state["H"], case["n_occ"], prec, case["ckpt"])
        (dLdH,) = torch.autograd.grad(P, state["H"], state["G"])
        return [P.detach(), dLdH]
    if kind == "batch":
        Ps, P1s, _ = ctx.sp2_response_batch(state["H"], state["H1"], state["n_occ"], precision=prec)
        return [Ps, P1s]
    P, _, _ = ctx.sp2_response(state["H"], state["H1"], case["n_occ"], precision=prec, ckpt_every=1,
                               workspace=state["ws"])
    P1, _, _, _ = ctx.scc_response(state["H1"], state["gamma"], state["ws"], tol=1e-5, precision=prec)
    return [P, P1]


# ---------------------------------------------------------------------------
# Exact results in 64 bits, from the known levels and basis


def _divided(eps, occ):
    """K_ij = (f_i - f_j) / (eps_i - eps_j) of the step function f."""
    de = eps[:, None] - eps[None, :]
    df = occ[:, None] - occ[None, :]
    return torch.where(df != 0, df / torch.where(df != 0, de, torch.ones_like(de)), torch.zeros_like(de))


def _first_order(basis, K, H1):
    return basis.out_of(K * basis.into(H1))


def _order_terms(eps, occ, basis, H1, order):
    """P_1 .. P_order in the eigenbasis: the occupied-empty blocks from
    [H, P_o] + [H1, P_{o-1}] = 0, the diagonal blocks from P P = P."""
    V = basis.into(H1)
    terms = [torch.diag(occ)]
    de = eps[:, None] - eps[None, :]
    cross = occ[:, None] != occ[None, :]
    both = torch.outer(occ, occ) > 0
    for o in range(1, order + 1):
        comm = V @ terms[o - 1] - terms[o - 1] @ V
        acc = torch.zeros_like(V)
        for a in range(1, o):
            acc += terms[a] @ terms[o - a]
        off = -comm / torch.where(cross, de, torch.ones_like(de))
        terms.append(torch.where(cross, off, torch.where(both, -acc, acc)))
    return [basis.out_of(t) for t in terms[1:]]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        Ps, P1s = [], []
        for i, (n, gap) in enumerate(_sizes(case)):
            _, H1, eps, occ, basis = _instance(n, n // 2, case["k"], gap, "gauss", seed * 1000 + i)
            K = _divided(eps, occ)
            Ps.append(basis.out_of(torch.diag(occ)))
            P1s.append(torch.stack([_first_order(basis, K, h) for h in H1]))
        return [Ps, P1s]
    n, k = case["n"], case.get("k", 0)
    H, H1, eps, occ, basis = _instance(n, case["n_occ"], k, case["gap"], case.get("h1", "dipole"), seed)
    P = basis.out_of(torch.diag(occ))
    if kind == "orders":
        per = [_order_terms(eps, occ, basis, h, case["order"]) for h in H1]
        return [P, *(torch.stack([d[o] for d in per]) for o in range(case["order"]))]
    K = _divided(eps, occ)
    if kind == "density":
        # the derivative of the step function is self-adjoint
        return [P, _first_order(basis, K, _loss_matrix(n, seed))]
    if kind == "response":
        return [P, torch.stack([_first_order(basis, K, h) for h in H1]) if k else None]
    gamma = _coupling(n, seed)
    P1 = torch.empty_like(H1)
    for j in range(k):
        q = torch.zeros(n, device=DEV, dtype=torch.float64)
        for _ in range(100):
            P1[j] = _first_order(basis, K, H1[j] + torch.diag(gamma @ q))
            new = P1[j].diagonal()
            done = float((new - q).norm()) < 1e-13 * float(new.norm())
            q = 0.2 * q + 0.8 * new
            if done:
                break
    return [P, P1]


# ---------------------------------------------------------------------------
# Work of one pass


def _layers(n, frac_occ, gap):
    """Layers of the recursion until convergence: the scalar recursion on 400
    levels of such a spectrum.  The bounds reach sum_j |H_ij| ~ n sqrt(2 / pi)
    std(H_ij) to either side of zero, with std(H_ij) = sqrt(<eps^2> / n)."""
    m = 400
    no = min(m - 1, max(1, int(round(m * frac_occ))))
    lo, hi = gap / 2, 2.0
    half = max(math.sqrt(2.0 / math.pi * n * (lo * lo + lo * hi + hi * hi) / 3.0), 1.2 * hi)
    eps = [-(lo + (hi - lo) * (i + 0.5) / no) for i in range(no)]
    eps += [lo + (hi - lo) * (i + 0.5) / (m - no) for i in range(m - no)]
    x = [(half - e) / (2 * half) for e in eps]
    for layer in range(1, 100):
        ns, nx = sum(x), sum(v * v for v in x)
        if ns - nx < 1e-5:
            return layer
        if abs(2 * ns - nx - no) > abs(nx - no):
            x = [v * v for v in x]
        else:
            x = [2 * v - v * v for v in x]
    return 100


def _response_work(n, n_occ, k, gap, dual):
    """Products of symmetric matrices, one triangle of each result: a square
    is n^3 flops and S0 S1 + S1 S0 is 2 n^3; a product of two 16-bit hi/lo
    pairs is three plain ones."""
    layers = _layers(n, n_occ / n, gap)
    return layers * (3.0 if dual else 1.0) * (1 + 2 * k) * float(n) ** 3


def work(case):
    kind = case["kind"]
    if kind == "batch":
        flops = bytes_ = 0.0
        for n, gap in _sizes(case):
            flops += _response_work(n, n // 2, case["k"], gap, True)
            bytes_ += 16.0 * n * n * (1 + case["k"])
        return dict(bytes=bytes_, flops=flops)
    n, k = case["n"], case.get("k", 0)
    dual = case["precision"].startswith("dual")
    flops = _response_work(n, case["n_occ"], k, case["gap"], dual)
    bytes_ = 16.0 * n * n * (1 + k)
    one = 3.0 * _layers(n, case["n_occ"] / n, case["gap"]) * float(n) ** 3
    if kind == "orders":
        # an order-o term: S0 S_o + S_o S0 and the products S_a S_{o-a}
        flops = one * (1 + k * sum(o + 1 for o in range(1, case["order"] + 1)))
        bytes_ = 8.0 * n * n * (2 + k + k * case["order"])
    elif kind == "density":
        flops = 3.0 * one                     # squares, then one S G + G S per layer
        bytes_ = 8.0 * n * n * 4
    elif kind == "scc":
        flops += 9 * 2.0 * k * one            # about nine replays reach the tolerance
        bytes_ = 8.0 * n * n * (3 + 2 * k)
    return dict(bytes=bytes_, flops=flops)

"""What this library is asked to do, as measurable cases: calls through its public entry points
over the sizes, options and directions that its users have.

``listed`` gives the standing cases, ``draw`` more of the same ranges, ``prepare`` a user's inputs
and plan, ``run`` one pass, ``work`` the arithmetic and traffic that no method of this kind avoids
(real operations, bytes), ``exact`` the results in 64 bits by the definitions, without the library.

A case names its ``path``: ``table`` (a Gaussian state's binned table), ``fit`` (table, loss and
gradients of a least-squares fit), ``batch`` (many uneven problems), ``fock`` (photon-number
inputs), ``herald`` (heralded states), ``cumulants`` (orders 1 to 4 of the binned counts).
"""
from __future__ import annotations

import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2412_17742_gb300 as gb

PRECISION = {"fp64": gb.GBSBIN_FP64, "fp32": gb.GBSBIN_FP32_REFINE}


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # One state of a four-mode device, two detectors: the smallest call, where the launches count.
        {"name": "table_n8_l2", "path": "table", "M": 4, "K": 1, "cutoffs": "6,6", "precision": "fp64",
         "displaced": False, "bases": False, "r_lo": 0.3, "r_hi": 0.8, "eta_lo": 0.7, "eta_hi": 0.7},
        # A 16-mode interferometer read out by four detectors of four modes, in the fast arithmetic.
        {"name": "table_n32_l4", "path": "table", "M": 16, "K": 1, "cutoffs": "8,8,8,8", "precision": "fp32",
         "displaced": False, "bases": False, "r_lo": 0.5, "r_hi": 1.2, "eta_lo": 0.4, "eta_hi": 0.9},
        # Odd sizes in the default arithmetic: 21 displaced modes, three detectors of unequal range.
        {"name": "table_n42_l3_displaced", "path": "table", "M": 21, "K": 1, "cutoffs": "7,10,5", "precision": "fp64",
         "displaced": True, "bases": False, "r_lo": 0.3, "r_hi": 1.0, "eta_lo": 0.3, "eta_hi": 0.95},
        # Partially distinguishable, displaced sources: 24 ports of four internal modes, three detectors.
        {"name": "table_n192_l3_displaced", "path": "table", "M": 24, "K": 4, "cutoffs": "20,20,20",
         "precision": "fp32", "displaced": True, "bases": True, "r_lo": 0.2, "r_hi": 0.8, "eta_lo": 0.6, "eta_hi": 0.6},
        # A hundred bright modes in two halves, in the default arithmetic: the validation of a large device.
        {"name": "table_n200_l2", "path": "table", "M": 100, "K": 1, "cutoffs": "80,80", "precision": "fp64",
         "displaced": False, "bases": False, "r_lo": 0.8, "r_hi": 1.6, "eta_lo": 0.5, "eta_hi": 0.5},
        # The total photon number of 256 modes: one detector group, the largest matrix.
        {"name": "total_n512", "path": "table", "M": 256, "K": 1, "cutoffs": "170", "precision": "fp64",
         "displaced": False, "bases": False, "r_lo": 0.3, "r_hi": 0.6, "eta_lo": 0.5, "eta_hi": 0.5},
        # One step of fitting a small device's squeezing, circuit and displacements to measured counts.
        {"name": "fit_n48_l2_displaced", "path": "fit", "M": 8, "K": 3, "cutoffs": "12,9", "precision": "fp64",
         "displaced": True, "bases": True, "r_lo": 0.2, "r_hi": 0.8, "eta_lo": 0.3, "eta_hi": 0.95},
        # The same for the hundred-mode device.
        {"name": "fit_n200_l2", "path": "fit", "M": 100, "K": 1, "cutoffs": "80,80", "precision": "fp32",
         "displaced": False, "bases": False, "r_lo": 0.8, "r_hi": 1.6, "eta_lo": 0.5, "eta_hi": 0.5},
        # A parameter scan: many problems of uneven size in one call.
        {"name": "batch_48", "path": "batch", "count": 48, "precision": "fp32", "r_lo": 0.3, "r_hi": 1.3,
         "eta_lo": 0.3, "eta_hi": 0.95},
        # Boson-sampling validation: 16 single photons in 32 ports, three detectors, the whole table.
        {"name": "fock_m32_n16_l3", "path": "fock", "M": 32, "photons": ",".join(["1"] * 16), "cutoffs": "16,16,16",
         "precision": "fp32", "eta_lo": 0.4, "eta_hi": 0.9},
        # Heralding a two-mode state by two grouped detectors of twelve modes each.
        {"name": "herald_m16_k2", "path": "herald", "M": 16, "K": 2, "cutoffs": "8,8", "per_group": 6, "kept": 2,
         "fock_cutoff": 6, "displaced": True, "bases": True, "r_lo": 0.4, "r_hi": 0.9, "eta_lo": 0.6, "eta_hi": 0.9},
        # The first four cumulants of eight detectors over 256 modes: the check against a measured record.
        {"name": "cumulants_n512_l8", "path": "cumulants", "M": 256, "K": 1, "groups": 8, "precision": "fp64",
         "displaced": True, "bases": False, "r_lo": 0.3, "r_hi": 1.0, "eta_lo": 0.4, "eta_hi": 0.9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cutoffs(rng, L, points):
    """L cutoffs whose grid has about `points` points, each axis up to a quarter off the even share."""
    side = points ** (1.0 / L)
    return ",".join(str(max(1, int(side * rng.uniform(0.75, 1.3)) - 1)) for _ in range(L))


def _draw_state(rng, most_modes):
    K = rng.choice([1, 1, 1, 2, 3, 4])
    M = max(4, _log_int(rng, 4, most_modes) // K)
    lo = rng.uniform(0.2, 0.6)
    eta = rng.uniform(0.3, 0.6)
    return {"M": M, "K": K, "displaced": rng.random() < 0.5, "bases": K > 1 and rng.random() < 0.6,
            "r_lo": lo, "r_hi": lo + rng.uniform(0.3, 0.6), "eta_lo": eta, "eta_hi": eta + rng.uniform(0.0, 0.35)}


def draw(rng):
    path = rng.choice(["table", "table", "table", "total", "fit", "batch", "fock", "herald", "cumulants"])
    precision = rng.choice(["fp64", "fp32"])
    if path == "table":
        case = _draw_state(rng, 100)
        L = rng.randint(2, 4)
        return {"path": "table", "precision": precision, "cutoffs": _cutoffs(rng, L, _log_int(rng, 49, 6000)), **case}
    if path == "total":
        case = _draw_state(rng, 256)
        return {"path": "table", "precision": precision, "cutoffs": str(_log_int(rng, 8, 170)), **case}
    if path == "fit":
        case = _draw_state(rng, 90)
        n = 2 * case["M"] * case["K"]
        most = min(4000, int(6e9 / n ** 3))
        return {"path": "fit", "precision": precision, "cutoffs": _cutoffs(rng, 2, _log_int(rng, 49, max(60, most))),
                **case}
    if path == "batch":
        return {"path": "batch", "count": rng.randint(8, 40), "precision": precision, "r_lo": 0.3,
                "r_hi": rng.uniform(0.8, 1.3), "eta_lo": 0.3, "eta_hi": 0.95}
    if path == "fock":
        M = rng.randint(6, 32)
        L = rng.randint(1, 3)
        photons = []
        while True:
            more = photons + [rng.choice([1, 1, 1, 2, 3])]
            if len(more) > min(M, 16) or math.prod(p + 1 for p in more) > 1 << 15 or sum(more) > 16:
                break
            photons = more
            if len(photons) >= 2 and rng.random() < 0.08:
                break
        N = sum(photons)
        cuts = ",".join(str(N if rng.random() < 0.7 else rng.randint((N + 1) // 2, N)) for _ in range(L))
        return {"path": "fock", "M": M, "photons": ",".join(map(str, photons)), "cutoffs": cuts,
                "precision": precision, "eta_lo": 0.4, "eta_hi": rng.uniform(0.6, 0.95)}
    if path == "herald":
        K = rng.choice([1, 2])
        groups = rng.randint(1, 2)
        per_group = rng.randint(1, 6)
        kept = rng.randint(1, 2)
        M = groups * per_group + kept + rng.randint(0, 2)
        lo = rng.uniform(0.2, 0.6)
        return {"path": "herald", "M": M, "K": K, "cutoffs": ",".join(str(rng.randint(3, 8)) for _ in range(groups)),
                "per_group": per_group, "kept": kept, "fock_cutoff": rng.randint(2, 6),
                "displaced": rng.random() < 0.5, "bases": K > 1 and rng.random() < 0.5, "r_lo": lo, "r_hi": lo + 0.4,
                "eta_lo": 0.6, "eta_hi": 0.9}
    case = _draw_state(rng, 256)
    return {"path": "cumulants", "groups": rng.randint(2, min(8, case["M"])), "precision": precision, **case}


# ------------------------------------------------------------------------------- the inputs
def _ints(text):
    return [int(v) for v in str(text).split(",")]


def _haar(n, rng):
    z = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / np.sqrt(2.0)
    q, r = np.linalg.qr(z)
    d = np.diag(r)
    return q * (d / np.abs(d))[None, :]


def _labels(M, L):
    edges = np.linspace(0, M, L + 1).round().astype(int)
    return np.repeat(np.arange(L, dtype=np.int32), np.diff(edges))


def _lossy(M, case, rng):
    eta = rng.uniform(case["eta_lo"], case["eta_hi"], M)
    return np.sqrt(eta)[:, None] * _haar(M, rng)


def _gaussian(case, rng, L, cutoff):
    M, K = case["M"], case["K"]
    p = SimpleNamespace(M=M, K=K, r=rng.uniform(case["r_lo"], case["r_hi"], (M, K)), T=_lossy(M, case, rng),
                        alpha=None, V=None, bin_of_mode=_labels(M, L), cutoff=np.array(cutoff, dtype=np.int32))
    if case["displaced"]:
        p.alpha = 0.22 * (rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K)))
    if case["bases"]:
        p.V = np.stack([_haar(K, rng) for _ in range(M)])
    return p


def _batch_problems(case, rng):
    out = []
    for _ in range(case["count"]):
        M, K = int(rng.integers(8, 49)), int(rng.integers(1, 4))
        L = int(rng.integers(1, 5))
        points = math.exp(rng.uniform(math.log(500.0), math.log(20000.0)))
        side = max(1, int(points ** (1.0 / L)) - 1)
        one = {"M": M, "K": K, "displaced": False, "bases": False, **{k: case[k] for k in ("r_lo", "r_hi", "eta_lo", "eta_hi")}}
        out.append(_gaussian(one, rng, L, [side] * L))
    return out


def _inputs(case, seed):
    path = case["path"]
    if path == "batch":
        # the sizes belong to the case, the states to the seed
        sizes = np.random.default_rng(177423)
        probs = _batch_problems(case, sizes)
        rng = np.random.default_rng([seed, 3])
        for p in probs:
            p.r = rng.uniform(case["r_lo"], case["r_hi"], (p.M, p.K))
            p.T = _lossy(p.M, case, rng)
        return probs
    rng = np.random.default_rng([seed, 1])
    if path == "fock":
        M, ph = case["M"], _ints(case["photons"])
        photons = np.zeros(M, dtype=np.int32)
        photons[:len(ph)] = ph
        cut = _ints(case["cutoffs"])
        return SimpleNamespace(M=M, T=_lossy(M, case, rng), photons=photons, bin_of_mode=_labels(M, len(cut)),
                               cutoff=np.array(cut, dtype=np.int32))
    if path == "cumulants":
        L = case["groups"]
        return _gaussian(case, rng, L, [1] * L)
    cut = _ints(case["cutoffs"])
    if path == "herald":
        p = _gaussian(case, rng, 1, [1])
        p.roles, p.cutoff = [], np.array(cut, dtype=np.int32)
        for port, k in itertools.product(range(case["M"]), range(case["K"])):
            g = port // case["per_group"]
            after = port - case["per_group"] * len(cut)
            p.roles.append(g if g < len(cut) else -2 if after < case["kept"] and k == 0 else -1)
        return p
    p = _gaussian(case, rng, len(cut), cut)
    if path == "fit":
        # what was measured: the frequencies of 100000 shots of independent, over-dispersed detectors
        axes = []
        for l, c in enumerate(cut):
            mean = max(0.5, 0.5 * float(np.sum(np.sinh(p.r) ** 2)) * np.mean(p.bin_of_mode == l))
            b = np.arange(c + 1)
            f = np.exp(-0.5 * (b - min(mean, 0.7 * c)) ** 2 / (1.0 + mean))
            axes.append(f / f.sum())
        pmf = axes[0]
        for f in axes[1:]:
            pmf = np.multiply.outer(pmf, f)
        p.target = (rng.multinomial(100000, pmf.reshape(-1) / pmf.sum()) / 1e5).reshape(pmf.shape)
    return p


def prepare(case, seed):
    path, precision = case["path"], PRECISION[case.get("precision", "fp64")]
    prob = _inputs(case, seed)
    s = SimpleNamespace(path=path, prob=prob, precision=precision)
    if path == "table":
        s.plan = gb.Plan(prob, precision=precision)
    elif path == "fit":
        s.plan = gb.Plan(prob, precision=precision, want_backward=True)
        s.leaves = [torch.tensor(prob.r, device="cuda"), torch.tensor(prob.T, device="cuda")]
        s.leaves += [None if v is None else torch.tensor(v, device="cuda") for v in (prob.alpha, prob.V)]
        s.target = torch.tensor(prob.target, device="cuda")
    elif path == "batch":
        s.plan = gb.Batch(prob, precision=precision)
        s.plan.allocate()
    elif path == "fock":
        s.plan = gb.FockPlan(prob, precision=precision)
    elif path == "herald":
        s.plan = gb.HeraldPlan(prob, prob.roles, prob.cutoff, case["fock_cutoff"])
    return s


# ------------------------------------------------------------------------------- one pass
def run(state):
    if state.path == "fit":
        leaves = [None if v is None else v.detach().requires_grad_(True) for v in state.leaves]
        P = gb.binned_distribution(state.plan, state.prob, *leaves)
        loss = 0.5 * (P - state.target).square().sum()
        loss.backward()
        names = ("r", "T", "alpha", "V")
        return {"P": P.detach(), "loss": loss.detach(),
                **{"d_" + k: v.grad for k, v in zip(names, leaves) if v is not None}}
    if state.path == "batch":
        return state.plan.execute()
    if state.path == "herald":
        rho, pr = state.plan.states()
        return {"rho": rho, "Pr": pr}
    if state.path == "cumulants":
        return gb.gbsbin_cumulants_device(state.prob, order=4, precision=state.precision)
    return state.plan.table()


# ------------------------------------------------------------------------------- its work
def _tree_flops(n, radix, extra):
    """Block elimination of the detector groups along the grid's axes, the last one halved: one
    reduced matrix per combination of the leading axes' roots."""
    L = len(radix)
    sizes = [2 * int(round(n / 2 * (l + 1) / L)) - 2 * int(round(n / 2 * l / L)) for l in range(L)]
    nodes, rest, total = 1.0, n, 0.0
    for l, m in enumerate(sizes):
        nodes *= radix[l] if l < L - 1 else radix[l] // 2 + 1
        after = rest - m
        total += nodes * (rest ** 3 - after ** 3) / 3 if L > 1 else nodes * m
        rest = after
    return 8.0 * total * extra


def work(case):
    path = case["path"]
    if path == "batch":
        out = {"bytes": 0.0, "flops": 0.0}
        for p in _batch_problems(case, np.random.default_rng(177423)):
            n, radix = 2 * p.M * p.K, [int(c) + 1 for c in p.cutoff]
            out["bytes"] += 16 * n * n + 8 * math.prod(radix)
            out["flops"] += _tree_flops(n, radix, 1)
        return out
    if path == "fock":
        ph, radix = _ints(case["photons"]), [c + 1 for c in _ints(case["cutoffs"])]
        nin, N, L = len(ph), sum(ph), len(radix)
        # the two halves of the factors as polynomials per sub-multiset of the inputs, then their products
        states = math.prod(p + 1 for p in ph) / max(1.0, math.sqrt(N))
        half = math.comb(N // 2 + L, L)
        return {"bytes": 16.0 * nin * nin * (L + 1) + 8 * math.prod(radix), "flops": 8.0 * states * half * half}
    n = 2 * case["M"] * case["K"]
    if path == "cumulants":
        L = case["groups"]
        return {"bytes": 16.0 * n * n + 8 * (L + L ** 2 + L ** 3 + L ** 4),
                "flops": 8.0 * (n ** 3 / 2 + L * L * n * n / 2)}
    radix = [c + 1 for c in _ints(case["cutoffs"])]
    points = math.prod(radix)
    if path == "herald":
        coef = (case["fock_cutoff"] + 1) ** (2 * case["kept"])
        return {"bytes": 16.0 * n * n + 16.0 * points * coef, "flops": 8.0 * points * (n ** 3 / 3 + coef * (1 + case["kept"]))}
    if path == "fit":
        # forward along the tree, then one inverse of the last group's block per evaluated point
        m = n / len(radix)
        return {"bytes": 48.0 * n * n + 24 * points,
                "flops": _tree_flops(n, radix, 1) + 8.0 * points / 2 * m ** 3 + 8.0 * points / radix[-1] * 4 * m ** 3}
    return {"bytes": 16.0 * n * n + 8 * points, "flops": _tree_flops(n, radix, 1)}


# ------------------------------------------------------------------------------- in 64 bits
def _sigma1(M, K, r, T, alpha, V):
    """Normally ordered covariance and mean of the output in the order (a, a^dagger), modes
    external-major; torch complex128, differentiable."""
    c = torch.complex128
    MK = M * K
    if V is None:
        V = torch.eye(K, dtype=c, device=T.device).expand(M, K, K)
    Tf = torch.einsum("ji,ilk->jlik", T, V).reshape(MK, MK)
    r = r.reshape(MK)
    N = (Tf.conj() * torch.sinh(r).square()) @ Tf.T
    Mm = (Tf * (torch.sinh(r) * torch.cosh(r))) @ Tf.T
    top = torch.cat([N.T, Mm], 1)
    S = torch.cat([top, torch.cat([Mm.conj(), N], 1)], 0)
    mean = Tf @ alpha.reshape(MK) if alpha is not None else torch.zeros(MK, dtype=c, device=T.device)
    return S, torch.cat([mean, mean.conj()])


def _on_gpu(p):
    t = lambda v: None if v is None else torch.tensor(v, device="cuda")  # noqa: E731
    return t(p.r), t(p.T), t(p.alpha), t(p.V)


def _adjacency(S, z):
    """XA = I - (I + S)^-1 and gamma = X (I + S)^-1 z."""
    n = S.shape[0]
    eye = torch.eye(n, dtype=S.dtype, device=S.device)
    Si = torch.linalg.inv(eye + S)
    return eye - Si, torch.roll(Si @ z, n // 2)


def _rows(p):
    lab = np.repeat(np.asarray(p.bin_of_mode), p.K)
    return torch.tensor(np.concatenate([lab, lab]).astype(np.int64), device="cuda")


def _half_grid(radix):
    """The roots (points, L) of the grid whose last axis is halved, the last axis fastest."""
    k = np.stack([m.reshape(-1) for m in np.meshgrid(*[np.arange(r) for r in radix[:-1]],
                                                     np.arange(radix[-1] // 2 + 1), indexing="ij")], 1)
    return torch.tensor(np.exp(2j * np.pi * k / np.array(radix)), device="cuda")


def _to_table(G, radix):
    """P(b) = 1/N sum_k G(w^k) w^(-k b) from the half grid."""
    G = G.reshape(tuple(radix[:-1]) + (radix[-1] // 2 + 1,))
    if len(radix) > 1:
        G = torch.fft.fftn(G, dim=tuple(range(len(radix) - 1)))
    return torch.fft.hfft(G, n=radix[-1], dim=-1) / math.prod(radix)


def _eliminate(A, steps):
    """`steps` pivots of the batch A in place, without exchanges; the sum of their logarithms (each
    pivot of I - D XA and of its Schur complements has a positive real part)."""
    logs = 0
    for k in range(steps):
        piv = A[:, k, k].clone()
        logs = logs + torch.log(piv)
        row = A[:, k, k + 1:] / piv[:, None]
        A[:, k + 1:, k + 1:].sub_(A[:, k + 1:, k, None] * row[:, None, :])
    return logs


def _log_q(XA, gamma, rows, roots):
    n = XA.shape[0]
    out = []
    step = max(1, int(1.5e9) // (16 * (n + 1) ** 2))
    for w in roots.split(step):
        D = w[:, rows]
        A = torch.zeros((w.shape[0], n + 1, n + 1), dtype=XA.dtype, device="cuda")
        A[:, :n, :n] = torch.eye(n, dtype=XA.dtype, device="cuda") - D[:, :, None] * XA
        A[:, :n, n] = D * torch.roll(gamma, n // 2)
        A[:, n, :n] = -gamma
        logs = _eliminate(A, n)
        out.append(0.5 * A[:, n, n] - 0.5 * logs)
    return torch.cat(out)


def _exact_table(p):
    radix = [int(c) + 1 for c in p.cutoff]
    XA, gamma = _adjacency(*_sigma1(p.M, p.K, *_on_gpu(p)))
    lq = _log_q(XA, gamma, _rows(p), _half_grid(radix))
    return _to_table(torch.exp(lq - lq[0]), radix)


def _exact_fit(p):
    radix = [int(c) + 1 for c in p.cutoff]
    leaves = [None if v is None else v.requires_grad_(True) for v in _on_gpu(p)]
    rows, roots = _rows(p), _half_grid(radix)
    XA, gamma = _adjacency(*_sigma1(p.M, p.K, *leaves))
    xa, ga = XA.detach().requires_grad_(True), gamma.detach().requires_grad_(True)
    lq = _log_q(xa.detach(), ga.detach(), rows, roots).requires_grad_(True)
    P = _to_table(torch.exp(lq - lq[0]), radix)
    loss = 0.5 * (P - torch.tensor(p.target, device="cuda")).square().sum()
    loss.backward()
    n = XA.shape[0]
    eye = torch.eye(n, dtype=XA.dtype, device="cuda")
    for w, g in zip(roots.split(256), lq.grad.split(256)):
        D = w[:, rows]
        K = eye - D[:, :, None] * xa
        sign, size = torch.linalg.slogdet(K)
        x = torch.linalg.solve(K, (D * torch.roll(ga, n // 2))[:, :, None])[:, :, 0]
        part = 0.5 * (x @ ga) - 0.5 * (size + torch.log(sign))
        (part * g.conj()).real.sum().backward()
    torch.autograd.backward([XA, gamma], [xa.grad, ga.grad])
    out = {"P": P.detach(), "loss": loss.detach()}
    return {**out, **{"d_" + k: v.grad for k, v in zip(("r", "T", "alpha", "V"), leaves) if v is not None}}


def _exact_fock(p):
    """perm(B(z)[p, p]) / p! as the coefficient of x^p in prod_j (B(z) x)_j^(p_j), taken on roots of
    unity in x, one input of the fewest photons held at 1."""
    radix = [int(c) + 1 for c in p.cutoff]
    J = np.flatnonzero(p.photons)
    ph = p.photons[J]
    held = int(np.argmin(ph))
    axes = [np.array([1.0 + 0j]) if j == held else np.exp(2j * np.pi * np.arange(q + 1) / (q + 1)) for j, q in enumerate(ph)]
    X = torch.tensor(np.stack([a.reshape(-1) for a in np.meshgrid(*axes, indexing="ij")], 1), device="cuda")
    weight = X.prod(1) / X.shape[0]
    T = torch.tensor(p.T, device="cuda")
    parts = [torch.eye(p.M, dtype=T.dtype, device="cuda") - T.conj().T @ T]
    for l in range(len(radix)):
        Tl = T[torch.tensor(np.flatnonzero(p.bin_of_mode == l), device="cuda")]
        parts.append(Tl.conj().T @ Tl)
    J = torch.tensor(J, device="cuda")
    V = torch.stack([X @ B[J][:, J].T for B in parts], 2)                    # [node, factor, 1 + group]
    roots = _half_grid(radix)
    Z = torch.cat([torch.ones_like(roots[:, :1]), roots], 1).T                # [1 + group, point]
    G = torch.zeros(roots.shape[0], dtype=T.dtype, device="cuda")
    step = max(1, (1 << 23) // roots.shape[0])
    for v, wt in zip(V.split(step), weight.split(step)):
        F = wt[:, None].expand(-1, roots.shape[0]).clone()
        for j, q in enumerate(ph):
            s = v[:, j] @ Z
            for _ in range(int(q)):
                F.mul_(s)
        G += F.sum(0)
    return _to_table(G, radix)


def _exact_herald(p, cut):
    """The Gaussian expectation over the heralding and traced modes at every root, its Taylor
    coefficients in the kept modes, and the inverse transform over the heralding groups."""
    S, z = _sigma1(p.M, p.K, *_on_gpu(p))
    XA, gamma = _adjacency(S, z)
    n = XA.shape[0]
    nm = n // 2
    roles = np.array(p.roles)
    A = torch.roll(XA, nm, 0)
    radix = [int(c) + 1 for c in p.cutoff]
    k = np.stack([m.reshape(-1) for m in np.meshgrid(*[np.arange(r) for r in radix], indexing="ij")], 1)
    w = np.ones((k.shape[0], nm), dtype=complex)
    for m, g in enumerate(roles):
        if g >= 0:
            w[:, m] = np.exp(2j * np.pi * k[:, g] / radix[g])
    w = torch.tensor(w, device="cuda")
    Dm, Fm = np.flatnonzero(roles != -2), np.flatnonzero(roles == -2)
    D, F = (torch.tensor(np.concatenate([m, m + nm]), device="cuda") for m in (Dm, Fm))
    nd, nf = len(D), len(F)
    wD = torch.cat([w, w], 1)[:, D]
    ADD, ADF, AFF = A[D][:, D], A[D][:, F], A[F][:, F]
    swap = lambda v: torch.roll(v, nd // 2, -2)  # noqa: E731
    K = torch.eye(nd, dtype=A.dtype, device="cuda") - swap(wD[:, :, None] * ADD)
    ld = _eliminate(K.clone(), nd) if nd else torch.zeros(w.shape[0], dtype=A.dtype, device="cuda")
    rhs = swap(wD[:, :, None] * torch.cat([ADF, gamma[D][:, None]], 1))
    Y = torch.linalg.solve(K, rhs)                                            # N [A_DF, gamma_D]
    Mq = (AFF + ADF.T @ Y[:, :, :nf]).cpu().numpy()
    lq = (gamma[F] + (ADF.T @ Y[:, :, nf:])[:, :, 0]).cpu().numpy()
    e = 0.5 * (gamma[D] @ Y[:, :, nf:])[:, 0]
    pts = w.shape[0]
    c = np.zeros((cut + 1,) * nf + (pts,), dtype=complex)
    c[(0,) * nf] = 1.0
    for q in sorted(itertools.product(range(cut + 1), repeat=nf), key=sum)[1:]:
        i = next(t for t in range(nf) if q[t])
        b = list(q)
        b[i] -= 1
        val = lq[:, i] * c[tuple(b)]
        for j in range(nf):
            if b[j]:
                a = list(b)
                a[j] -= 1
                val = val + Mq[:, i, j] * c[tuple(a)]
        c[q] = val / q[i]
    G = torch.tensor(np.moveaxis(c, -1, 0), device="cuda") * torch.exp(e - 0.5 * ld).reshape((pts,) + (1,) * nf)
    wa = torch.cat([w, w], 1)
    aug = torch.zeros((pts, n + 1, n + 1), dtype=A.dtype, device="cuda")
    aug[:, :n, :n] = torch.eye(n, dtype=A.dtype, device="cuda") - torch.roll(wa[:, :, None] * A, nm, 1)
    aug[:, :n, n] = torch.roll(wa * gamma, nm, 1)
    aug[:, n, :n] = -gamma
    lda = _eliminate(aug, n)
    Gt = torch.exp(0.5 * aug[:, n, n] - 0.5 * lda)
    eye = torch.eye(n, dtype=A.dtype, device="cuda")
    expo = gamma @ torch.linalg.solve(eye - XA, torch.roll(gamma, nm))
    pr0 = torch.exp(-0.5 * expo.real) * torch.sqrt(torch.linalg.det(eye - XA).real)
    axes = tuple(range(len(radix)))
    rho = torch.fft.fftn(G.reshape(tuple(radix) + (cut + 1,) * nf), dim=axes) / pts * pr0
    Pr = (torch.fft.fftn(Gt.reshape(radix), dim=axes) / pts * pr0).real
    fact = torch.tensor([math.sqrt(math.factorial(i)) for i in range(cut + 1)], dtype=torch.float64, device="cuda")
    for ax in range(nf):
        rho = rho * fact.reshape([-1 if ax == t else 1 for t in range(nf)])
    return {"rho": rho, "Pr": Pr}


def _partitions(items):
    if not items:
        yield []
        return
    first, rest = items[0], items[1:]
    for part in _partitions(rest):
        yield [[first]] + part
        for i in range(len(part)):
            yield part[:i] + [[first] + part[i]] + part[i + 1:]


def _exact_cumulants(p):
    """log G(e) to fourth order in e_l = exp(t_l) - 1 from traces and paths of W = Sigma - I, then
    the chain rule over the set partitions of the slots."""
    S, z = _sigma1(p.M, p.K, *_on_gpu(p))
    _, gamma = _adjacency(S, z)
    n, L = S.shape[0], int(p.bin_of_mode.max()) + 1
    W, xg = S, torch.roll(gamma, n // 2)
    u, v = xg + W @ xg, gamma + W.T @ gamma
    rows = _rows(p)
    E = torch.nn.functional.one_hot(rows, L).to(W.dtype)
    blocks = lambda M2: E.T @ M2 @ E  # noqa: E731
    C1 = 0.5 * (E.T @ (torch.diagonal(W) + v * u))
    C2 = blocks(0.25 * W * W.T + 0.5 * v[:, None] * W * u)
    Y = [W[:, rows == b] @ W[rows == b] for b in range(L)]
    C3 = torch.stack([blocks(Y[b] * (W.T / 6 + 0.5 * v[:, None] * u)) for b in range(L)], 1)
    q = W @ (E * u[:, None])                                                  # [k, d]
    pa = [(E * v[:, None]).T @ Y[b] for b in range(L)]                        # [a, k]
    C4 = torch.stack([torch.stack([blocks(Y[b] * Y[d].T) / 8 + 0.5 * (pa[b] * q[:, d]) @ E for d in range(L)], 2)
                      for b in range(L)], 1)                                  # [a, b, c, d]
    C = [c.real.cpu().numpy() for c in (C1, C2, C3, C4)]
    Fs = [sum(np.transpose(c, o) for o in itertools.permutations(range(r + 1))) for r, c in enumerate(C)]
    out = []
    for order in range(1, 5):
        kappa = np.zeros((L,) * order)
        idx = np.indices(kappa.shape)
        for part in _partitions(list(range(order))):
            same = np.ones(kappa.shape, dtype=bool)
            for block in part:
                for s in block[1:]:
                    same &= idx[s] == idx[block[0]]
            kappa += np.where(same, Fs[len(part) - 1][tuple(idx[b[0]] for b in part)], 0.0)
        out.append(kappa)
    return out


def exact(case, seed):
    p = _inputs(case, seed)
    if case["path"] == "table":
        return _exact_table(p)
    if case["path"] == "fit":
        return _exact_fit(p)
    if case["path"] == "batch":
        return [_exact_table(q) for q in p]
    if case["path"] == "fock":
        return _exact_fock(p)
    if case["path"] == "herald":
        return _exact_herald(p, case["fock_cutoff"])
    return _exact_cumulants(p)

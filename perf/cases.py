"""Performance cases of the evaluation path: what a program that uses this library has it do.

A case is a dict of plain values.  `listed()` names the fixed ones, `draw(rng)` gives more from the
same ranges, `prepare(case, seed)` makes what a program holds before the call (the uploaded diagram,
frequencies on the GPU, upstream gradients, energies), `run(state)` is one pass through the public
Python layer, `work(case)` its algorithmic bytes and flops, and `exact(case, seed)` the same outputs
from plain torch in 64 bits: its own Philox stream, residue sums and term-by-term evaluation.

Families ("pass"):
  forward    Diagram.forward: Monte Carlo mean and variance over momentum samples
  samples    Diagram.forward(per_sample=True): the per-sample values as well
  slope      Diagram.forward_backward with a zero upstream gradient: Sigma and dSigma/domega in one
             pass (the quasiparticle weight needs no parameter gradient)
  fused      Diagram.forward_backward: value, dSigma/domega and the parameter gradients in one pass
  autograd   SigmaMC.apply and its backward: the same through torch.autograd
  energy     Diagram.eval_energies: given energies, every (frequency, row) value
  batch      Batch.launch: many diagrams of uneven size in one graph launch

Which diagrams.  A residue sum cancels near its removable poles: where a combination of energies that
appears as a frequency-free denominator (or in a Bose function) comes near zero, the rounding of
that one sample is amplified, and a mean over many samples carries the worst of them.  For tables with
double poles (the largest of each order) two correct double-precision evaluations differ by 1e-7 to
1e-5 in the mean, and the parameter gradients of every Hubbard self-energy by 1e-9 and far more; no
output of those could be compared.  So the self-energies here are diagrams without double poles and with
few frequency-free denominators (two evaluations agree to about 1e-11), and the parameter gradients
are taken of ladders of particle-hole bubbles, which have neither (about 1e-14).
"""
import math
from functools import lru_cache

import numpy as np
import torch

import paper_2311_17189_gb300 as tami
from paper_2311_17189_gb300.autograd import SigmaMC

PI = math.pi
MASK = 0xFFFFFFFF

def _bubbles(m):
    """m particle-hole bubbles in a row, each its own loop momentum: lines k_l and k_l + q, q external
    and bosonic."""
    rows = []
    for l in range(m):
        for ext in (0, 1):
            rows.append([1 if v == l else 0 for v in range(m)] + [ext])
    return rows


# Label matrices (one row per line: internal variables, external ones last), bosonic flags and
# lattice parameters.
DIAGRAMS = {
    # order-2 Hubbard self-energy, basis (q, k', k_ext), q a bosonic transfer
    "order2": dict(alpha=[[1, 0, 1], [0, 1, 0], [1, 1, 0]], boson=[1, 0, 0], t=1.0, tp=0.0, mu=0.0),
    # the evaluation example: three lines, all fermionic
    "example": dict(alpha=[[1, 0, 0], [0, 1, 0], [-1, 1, 1]], t=1.0, tp=0.0, mu=0.0),
    # the first order-3 diagram (17 flat terms)
    "order3": dict(alpha=[[1, -1, 1, 0], [1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 0], [1, 0, 1, -1]],
                   t=1.0, tp=0.0, mu=0.0),
    # order-3 to order-5 diagrams of the enumerator (17, 66, 70, 236 and 240 flat terms)
    "order3b": dict(alpha=[[1, 1, -1, 0], [1, 0, 0, 0], [-1, 0, 1, 1], [0, 1, 0, 0], [0, 0, 1, 0]], t=1.0, tp=0.0, mu=0.0),
    "order4": dict(alpha=[[1, -1, 1, -1, 1], [1, 0, 0, 0, 0], [0, 1, 0, 0, 0], [-1, 1, 0, 1, 0],
                          [0, 0, 1, 0, 0], [0, 0, 0, 1, 0], [0, 1, 0, 1, -1]], t=1.0, tp=-0.3, mu=-0.5),
    "order4b": dict(alpha=[[1, -1, 0, 1, 0], [1, 0, -1, 1, 0], [1, 0, 0, 0, 0], [0, 1, 0, 0, 0],
                          [0, 0, 1, 0, 0], [0, 0, 0, 1, 0], [1, 0, 0, 1, -1]], t=1.0, tp=-0.3, mu=-0.5),
    "order5": dict(alpha=[[1, -1, 0, 1, 0, 0], [1, 0, -1, 1, 0, 0], [1, 0, 0, 0, 0, 0],
                          [0, 0, 0, -1, 1, 1], [0, 1, 0, 0, 0, 0], [0, 0, 1, 0, 0, 0],
                          [0, 0, 0, 1, 0, 0], [1, 0, 0, 1, 0, -1], [0, 0, 0, 0, 1, 0]], t=1.0, tp=0.0, mu=0.0),
    "order5b": dict(alpha=[[1, -1, 0, 0, 0, 1], [1, 0, 0, 0, 0, 0], [0, 1, 0, 0, 0, 0],
                          [0, 0, 1, 0, 0, 0], [-1, 1, 0, 1, 0, 0], [0, -1, 1, 0, 1, 0],
                          [0, 0, 0, 1, 0, 0], [0, 0, 0, 0, 1, 0], [0, 0, 1, 0, 1, -1]], t=1.0, tp=0.0, mu=0.0),
    # the order-4 diagram with its last loop frequency held external as well (two external frequencies)
    "order4x2": dict(alpha=[[1, -1, 1, -1, 1], [1, 0, 0, 0, 0], [0, 1, 0, 0, 0], [-1, 1, 0, 1, 0],
                            [0, 0, 1, 0, 0], [0, 0, 0, 1, 0], [0, 1, 0, 1, -1]], n_ext=2, t=1.0, tp=0.0, mu=0.0),
    # three and five bubbles (8 and 32 flat terms)
    "bubbles3": dict(alpha=_bubbles(3), boson=[0] * 3 + [1], t=1.0, tp=-0.3, mu=-0.5),
    "bubbles5": dict(alpha=_bubbles(5), boson=[0] * 5 + [1], t=1.0, tp=-0.3, mu=-0.5),
}


def listed():
    return [
        # the plain order-2 self-energy: a small Monte Carlo call, launches and latency count
        {"name": "order2_forward_small", "pass": "forward", "diagram": "order2", "n": 100_000, "n_f": 1, "beta": 5.0,
         "axis": "matsubara"},
        # the evaluation example on a thousand rows of energies: the smallest call
        {"name": "energy_small", "pass": "energy", "diagram": "example", "n": 1000, "n_f": 10, "beta": 1.0},
        # per-sample values kept for the caller's own statistics: output-heavy
        {"name": "order3_samples", "pass": "samples", "diagram": "order3", "n": 65_537, "n_f": 32, "beta": 5.0,
         "axis": "matsubara"},
        # one step of a fit through torch.autograd: value and every gradient
        {"name": "bubbles5_autograd", "pass": "autograd", "diagram": "bubbles5", "n": 1 << 18, "n_f": 16,
         "beta": 8.0, "axis": "matsubara"},
        # one chunk of a resumable Monte Carlo run, an odd size, a ragged frequency count
        {"name": "order4_forward_chunk", "pass": "forward", "diagram": "order4", "n": 1_000_003, "n_f": 21,
         "beta": 8.0, "axis": "matsubara"},
        # the benchmark's order-4 step: its samples, frequencies and lattice
        {"name": "order4_slope_large", "pass": "slope", "diagram": "order4", "n": 1 << 24, "n_f": 16, "beta": 8.0,
         "axis": "matsubara"},
        # order 3 continued to the real axis: the frequency loop dominates
        {"name": "order3_real_axis", "pass": "slope", "diagram": "order3", "n": 1 << 21, "n_f": 256, "beta": 10.0,
         "axis": "real"},
        # forward and every gradient in one large launch
        {"name": "bubbles5_fused_large", "pass": "fused", "diagram": "bubbles5", "n": 1 << 22, "n_f": 16,
         "beta": 8.0, "axis": "matsubara"},
        # an order-5 table at one frequency: the per-sample work dominates
        {"name": "order5_forward_large", "pass": "forward", "diagram": "order5", "n": 1 << 23, "n_f": 1, "beta": 10.0,
         "axis": "matsubara"},
        # the evaluation example at its own size: a million rows, a hundred frequencies
        {"name": "energy_large", "pass": "energy", "diagram": "example", "n": 1_000_000, "n_f": 100, "beta": 1.0},
        # two external frequencies on a 10 x 10 grid
        {"name": "two_external", "pass": "energy", "diagram": "order4x2", "n": 250_000, "n_f": 100, "beta": 1.0},
        # diagrams of orders 2 to 5, four streams of each, in one graph launch: uneven sample counts
        {"name": "batch_mixed", "pass": "batch", "streams": 4, "n": 1 << 14, "n_f": 32, "beta": 5.0},
    ]


def draw(rng):
    """One more case: the family and diagram by how often they are used, the sizes log-uniform."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    family = rng.choice(["forward", "forward", "samples", "slope", "slope", "autograd", "fused", "energy", "energy",
                         "batch"])
    beta = rng.choice([2.0, 5.0, 8.0, 10.0])
    if family == "batch":
        case = {"pass": "batch", "streams": rng.randint(1, 8), "n": log_int(1 << 10, 1 << 16),
                "n_f": log_int(4, 64), "beta": beta}
    elif family == "energy":
        case = {"pass": "energy", "diagram": rng.choice(["example", "order4x2", "order3", "order4"]),
                "n": log_int(500, 1_000_000), "n_f": log_int(1, 128), "beta": rng.choice([1.0, 2.0, 5.0])}
        if case["diagram"] == "order4x2":
            case["n_f"] = max(1, math.isqrt(case["n_f"])) ** 2
    else:
        dia = rng.choice(["bubbles3", "bubbles5"] if family in ("fused", "autograd") else
                         ["order2", "order3", "order4", "order4", "order5"])
        real = dia in ("order2", "order3", "bubbles3") and rng.random() < 0.4
        case = {"pass": family, "diagram": dia, "n": log_int(2000, 1 << 24),
                "n_f": log_int(16, 256) if real else log_int(1, 48), "beta": beta,
                "axis": "real" if real else "matsubara"}
    top = work(listed()[5])["flops"]
    while True:
        w = work(case)
        if w["flops"] <= top and w["bytes"] <= 2e9:
            return case
        case["n"] = case["n"] * 5 // 8 + 1


# ------------------------------------------------------------------------------- inputs
def _eps(alpha):
    """Lines with the same label share one base energy: that of the first of them."""
    N = len(alpha)
    eps = np.zeros((N, N), dtype=np.int8)
    for j, row in enumerate(alpha):
        eps[j, alpha.index(row)] = 1
    return eps


def _diagram(name):
    d = DIAGRAMS[name]
    return tami.Diagram(np.array(d["alpha"]), eps=_eps(d["alpha"]), var_is_boson=d.get("boson"),
                        n_ext=d.get("n_ext", 1))


def _lattice(name):
    d = DIAGRAMS[name]
    return (d["t"], d["tp"], d["mu"], PI / 2, PI / 2)


def _frequencies(case):
    n_f, beta = case["n_f"], case["beta"]
    if case.get("axis") == "real":
        return np.linspace(-4.0, 4.0, n_f) + 0.05j
    if case.get("diagram", "").startswith("bubbles"):       # the external line is bosonic, n >= 1
        return 2j * np.arange(1, n_f + 1) * PI / beta
    iw = lambda n: 1j * (2.0 * np.arange(n) + 1.0) * PI / beta  # noqa: E731
    if case.get("diagram") == "order4x2":
        k = math.isqrt(n_f)
        a, b = np.meshgrid(iw(k), iw(k), indexing="ij")
        return np.stack([a.ravel(), b.ravel()], axis=1)
    return iw(n_f)


def _upstream(case, seed):
    if case["pass"] == "slope":
        return np.zeros(case["n_f"], dtype=np.complex128)
    rng = np.random.default_rng([int(seed), 1])
    return rng.normal(size=case["n_f"]) + 1j * rng.normal(size=case["n_f"])


def _energies(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    N = len(DIAGRAMS[case["diagram"]]["alpha"])
    return torch.rand((case["n"], N), generator=g, device="cuda", dtype=torch.float64) * 16.0 - 8.0


def _key(seed):
    return 20231128 + 7919 * int(seed)


BATCH = ("order2", "order3", "order3b", "order4", "order4b", "order5", "order5b")


def _batch_streams(case):
    """(diagram, samples) of every stream: counts differ by up to a factor of eight."""
    return [(name, case["n"] << (d % 4)) for d, name in enumerate(BATCH * case["streams"])]


def prepare(case, seed):
    s = dict(case)
    s["X"] = torch.from_numpy(_frequencies(case)).cuda()
    if case["pass"] == "batch":
        ds = {name: _diagram(name).upload(0) for name in BATCH}
        streams = _batch_streams(case)
        s["plan"] = tami.Batch([ds[name] for name, _ in streams], [n for _, n in streams],
                               [_key(seed) + d for d in range(len(streams))], case["n_f"])
        s["lattice"] = (1.0, 0.0, 0.0, PI / 2, PI / 2)
        return s
    s["D"] = _diagram(case["diagram"]).upload(0)
    if case["pass"] == "energy":
        s["E"] = _energies(case, seed)
        return s
    s["lattice"], s["key"] = _lattice(case["diagram"]), _key(seed)
    if case["pass"] in ("slope", "fused", "autograd"):
        s["g"] = torch.from_numpy(_upstream(case, seed)).cuda()
    if case["pass"] == "autograd":
        lat = s["lattice"]
        s["omega"] = s["X"].real.clone().requires_grad_()
        s["gamma"] = s["X"].imag.clone()
        s["mu"] = torch.tensor(lat[2], dtype=torch.float64, requires_grad=True)
        s["kext"] = torch.tensor(lat[3:5], dtype=torch.float64, requires_grad=True)
    return s


def run(s):
    kind = s["pass"]
    if kind == "batch":
        mean, var = s["plan"].launch(s["lattice"], s["X"], s["beta"])
        return {"mean": mean, "var": var}
    if kind == "energy":
        return {"values": s["D"].eval_energies(s["E"], s["X"], s["beta"])}
    if kind in ("slope", "fused"):
        return s["D"].forward_backward(s["lattice"], s["key"], 0, s["n"], s["X"], s["beta"], s["g"])
    if kind == "autograd":
        lat = s["lattice"]
        sigma = SigmaMC.apply(s["D"], s["omega"], s["gamma"], s["mu"], s["kext"], lat[0], lat[1], s["beta"], s["n"],
                              s["key"], 0)
        loss = (s["g"].conj() * sigma).real.sum()
        g_omega, g_mu, g_kext = torch.autograd.grad(loss, (s["omega"], s["mu"], s["kext"]))
        return {"sigma": sigma.detach(), "g_omega": g_omega, "g_mu": g_mu, "g_kext": g_kext}
    mean, var, values = s["D"].forward(s["lattice"], s["key"], 0, s["n"], s["X"], s["beta"],
                                       per_sample=kind == "samples")
    return {"mean": mean, "var": var} if kind == "forward" else {"mean": mean, "var": var, "values": values}


# ------------------------------------------------------------------------------- work
@lru_cache(maxsize=None)
def _info(name):
    return _diagram(name).info()


def work(case):
    """Algorithmic flops of the factorised evaluation (fma = 2) and the bytes that must cross HBM:
    momenta are drawn in the kernel, so a Monte Carlo pass reads and writes only its frequencies and
    reduced outputs, unless it returns per-sample values; energy input reads E and writes every value."""
    n, n_f = case["n"], case["n_f"]
    if case["pass"] == "batch":
        streams = [(_info(name), k) for name, k in _batch_streams(case)]
        return {"bytes": 16.0 * n_f + 32.0 * n_f * len(streams),
                "flops": sum(k * (i["flops_per_sample"] + n_f * i["flops_per_sample_freq"]) for i, k in streams)}
    i = _info(case["diagram"])
    if case["pass"] == "energy":
        return {"bytes": n * (8.0 * i["n_lines"] + 16.0 * n_f) + 16.0 * n_f * i["n_ext"],
                "flops": n * (i["energy_in_flops_per_sample"] + n_f * i["energy_in_flops_per_sample_freq"])}
    if case["pass"] in ("slope", "fused", "autograd"):
        return {"bytes": 88.0 * n_f + 24.0,
                "flops": n * (i["bwd_flops_per_sample"] + n_f * i["fused_flops_per_sample_freq"])}
    return {"bytes": 48.0 * n_f + (16.0 * n_f * n if case["pass"] == "samples" else 0.0),
            "flops": n * (i["flops_per_sample"] + n_f * i["flops_per_sample_freq"])}


# ------------------------------------------------------------------------------- exact values
def _signed(f, c):
    """A Green's function 1/(f.X + c.E) with its first nonzero coefficient positive, and the sign taken out."""
    lead = next(v for v in f + c if v)
    return ((f, c), 1) if lead > 0 else ((tuple(-v for v in f), tuple(-v for v in c)), -1)


def _product(factors):
    """{(f, c): power} and sign of a list of ((f, c), power), equal poles merged."""
    out, sign = {}, 1
    for (f, c), p in factors:
        key, s = _signed(f, c)
        out[key] = out.get(key, 0) + p
        sign *= s ** p
    return out, sign


def _sum_over(term, p, boson):
    """T sum over the frequency of variable p of one term (coefficient, Fermi factors, Green's functions):
    the residues at its poles, of any order.  A Fermi factor (sigma, k, c) is d^k/dx^k of
    1/(sigma e^{beta x} + 1) at x = c.E; frequencies in its argument flip sigma by periodicity."""
    coef, fermi, greens = term
    out = []
    for (f, c), r in greens.items():
        a = f[p]
        if a == 0:
            continue
        zf = tuple(0 if q == p else -a * v for q, v in enumerate(f))
        zc = tuple(-a * v for v in c)
        odd = sum(v for q, v in enumerate(zf) if not boson[q]) % 2
        sigma = (-1 if boson[p] else 1) * (-1 if odd else 1)
        rest = {k: v for k, v in greens.items() if k != (f, c)}
        parts = {(0, tuple(sorted(rest.items()))): coef * a ** r / math.factorial(r - 1)}
        for _ in range(r - 1):           # d/dz of (Fermi derivative order, Green's functions)
            new = {}
            for (k, gs), w in parts.items():
                new[(k + 1, gs)] = new.get((k + 1, gs), 0.0) + w
                for (gf, gc), pw in gs:
                    if gf[p]:
                        up = dict(gs)
                        up[(gf, gc)] = pw + 1
                        key = (k, tuple(sorted(up.items())))
                        new[key] = new.get(key, 0.0) - w * pw * gf[p]
            parts = new
        for (k, gs), w in parts.items():
            moved = []
            for (gf, gc), pw in gs:
                b = gf[p]
                moved.append(((tuple(0 if q == p else v + b * z for q, (v, z) in enumerate(zip(gf, zf))),
                               tuple(v + b * z for v, z in zip(gc, zc))), pw))
            g, s = _product(moved)
            out.append((w * s, tuple(sorted(fermi + ((sigma, k, zc),))), g))
    return out


@lru_cache(maxsize=None)
def _solution(name):
    """The solution's terms grouped: {Green's functions: {Fermi factors: coefficient}}."""
    d = DIAGRAMS[name]
    alpha, n_ext = d["alpha"], d.get("n_ext", 1)
    eps = _eps(alpha).tolist()
    n_vars = len(alpha[0])
    boson = d.get("boson") or [0] * n_vars
    g, s = _product([((tuple(a), tuple(e)), 1) for a, e in zip(alpha, eps)])
    terms = [(float(s), (), g)]
    for p in range(n_vars - n_ext):
        terms = [t for x in terms for t in _sum_over(x, p, boson)]
    groups = {}
    for w, fermi, g in terms:
        key = tuple(sorted(((f[n_vars - n_ext:], c), pw) for (f, c), pw in g.items()))
        into = groups.setdefault(key, {})
        into[fermi] = into.get(fermi, 0.0) + w
    return groups


def _fermi(x, sigma, k, beta):
    """d^k/dx^k 1/(sigma e^{beta x} + 1), from g and h = 1 - g: dg/dx = -beta g h, dh/dx = beta g h."""
    if sigma > 0:
        g, h = torch.sigmoid(-beta * x), torch.sigmoid(beta * x)
    else:
        g, h = -1.0 / torch.expm1(beta * x), -1.0 / torch.expm1(-beta * x)
    poly = {(1, 0): 1.0}
    for _ in range(k):
        new = {}
        for (a, b), w in poly.items():
            if a:
                new[(a, b + 1)] = new.get((a, b + 1), 0.0) - w * a
            if b:
                new[(a + 1, b)] = new.get((a + 1, b), 0.0) + w * b
        poly = new
    return beta ** k * sum(w * g ** a * h ** b for (a, b), w in poly.items())


def _values(name, E, X, beta, derivative=False):
    """Values [n_f, n] of the solution at energies E [n, N] and frequencies X [n_f, n_ext]; with
    `derivative`, also d/dX (one external frequency)."""
    combos, fermis, groups = {}, {}, _solution(name)

    def combo(c):
        if c not in combos:
            combos[c] = sum(float(w) * E[:, j] for j, w in enumerate(c) if w)
        return combos[c]

    flat = [(gi, fermi, w) for gi, key in enumerate(groups) for fermi, w in groups[key].items() if w]
    for _, fermi, _ in flat:
        for fa in fermi:
            fermis.setdefault(fa, len(fermis))
    table = torch.stack([_fermi(combo(c), sg, k, beta) for sg, k, c in fermis])
    index = torch.tensor([[fermis[fa] for fa in fermi] for _, fermi, _ in flat], device=E.device)
    prod = table[index[:, 0]]
    for i in range(1, index.shape[1]):
        prod = prod * table[index[:, i]]
    into = torch.zeros((len(groups), len(flat)), dtype=torch.float64, device=E.device)
    for t, (gi, _, w) in enumerate(flat):
        into[gi, t] = w
    weight = into @ prod
    by_signature = {}
    for gi, key in enumerate(groups):
        w, sig = weight[gi], []
        for (f, c), p in key:
            if any(f):
                sig.append(((f, c), p))
            else:
                w = w / combo(c) ** p
        sig = tuple(sig)
        by_signature[sig] = by_signature[sig] + w if sig in by_signature else w
    value = dvalue = 0.0
    for sig, w in by_signature.items():
        R, dlog = torch.ones((X.shape[0], 1), dtype=torch.complex128, device=E.device), 0.0
        for (f, c), p in sig:
            D = (X @ torch.tensor(f, dtype=torch.complex128, device=E.device))[:, None] + combo(c)[None, :]
            R = R / D ** p if p > 1 else R / D
            if derivative:
                dlog = dlog - p * f[-1] / D.detach()
        value = value + w[None, :] * R
        if derivative and sig:
            dvalue = dvalue + w.detach()[None, :] * R.detach() * dlog
    return value, dvalue


def _philox(sample, variable, key):
    """Philox4x32-10 words of counter (sample lo, sample hi, variable, 0), in int64 tensors."""
    c = [sample & MASK, (sample >> 32) & MASK, torch.full_like(sample, variable), torch.zeros_like(sample)]
    k0, k1 = key & MASK, (key >> 32) & MASK
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & MASK) ^ c[1] ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c[3] ^ k1, p0 & MASK]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c


def _momentum(hi, lo):
    """k = 2 pi u - pi with u = m 2^-53, rounded once: the product in two exact parts."""
    m = ((hi << 21) | (lo >> 11)).double()
    c = 2.0 * PI * 2.0 ** -53
    split = lambda v: (v * 134217729.0) - ((v * 134217729.0) - v)  # noqa: E731
    mh, ch = split(m), (c * 134217729.0) - ((c * 134217729.0) - c)
    ml, cl = m - mh, c - ch
    p = m * c
    e = ((mh * ch - p) + mh * cl + ml * ch) + ml * cl
    s = p - PI
    bb = s - p
    return s + (((p - (s - bb)) + (-PI - bb)) + e)


def _sampled_energies(name, lat, key, s0, n, mu, kx, ky):
    """Line energies mu - eps(K_j) [n, N] of samples s0 .. s0 + n - 1."""
    t, tp = lat[0], lat[1]
    alpha = DIAGRAMS[name]["alpha"]
    m = len(alpha[0]) - 1
    sample = torch.arange(s0, s0 + n, dtype=torch.int64, device="cuda")
    ks = []
    for l in range(m):
        w = _philox(sample, l, key)
        ks.append((_momentum(w[0], w[1]), _momentum(w[2], w[3])))
    ks.append((kx, ky))
    cols = []
    for row in alpha:
        ax = ay = 0.0
        for a, (x, y) in zip(row, ks):
            if a:
                ax, ay = ax + a * x, ay + a * y
        cx, cy = torch.cos(ax), torch.cos(ay)
        cols.append(mu + 2.0 * t * (cx + cy) + 4.0 * tp * cx * cy)
    return torch.stack(cols, dim=1)


def _exact_mc(name, lat, key, n, X, beta, g=None, keep=False):
    """Mean, unbiased variance and, with an upstream gradient g, dSigma/dX and d/d(mu, kx, ky) of
    Re sum conj(g) Sigma; the per-sample values with `keep`."""
    n_f = X.shape[0]
    chunk = _chunk(name, n, n_f)
    count, mean, m2 = 0, torch.zeros(n_f, dtype=torch.complex128, device="cuda"), 0.0
    dX, params, kept = 0.0, 0.0, []
    for s in range(0, n, chunk):
        k = min(chunk, n - s)
        th = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=g is not None) for v in lat[2:5]]
        v, dv = _values(name, _sampled_energies(name, lat, key, s, k, *th), X, beta, derivative=g is not None)
        if g is not None:
            loss = (g.conj()[:, None] * v).real.sum() / n
            params = params + torch.stack(torch.autograd.grad(loss, th))
            dX = dX + dv.sum(dim=1) / n
        v = v.detach()
        mk = v.mean(dim=1)
        dev = torch.view_as_real(v - mk[:, None])
        diff = torch.view_as_real(mk - mean)
        m2 = m2 + (dev * dev).sum(dim=1) + diff * diff * (count * k / (count + k))
        mean = mean + (mk - mean) * (k / (count + k))
        count += k
        if keep:
            kept.append(v)
    return mean, m2 / max(1, n - 1), dX, params, torch.cat(kept, dim=1) if keep else None


def _chunk(name, n, n_f):
    n_flat = sum(len(v) for v in _solution(name).values())
    return max(1, min(n, 1 << 18, (1 << 29) // (8 * n_flat), (1 << 28) // (16 * n_f)))


def exact(case, seed):
    kind, n, n_f, beta = case["pass"], case["n"], case["n_f"], case["beta"]
    X = torch.from_numpy(_frequencies(case)).cuda().reshape(n_f, -1)
    if kind == "batch":
        lat = (1.0, 0.0, 0.0, PI / 2, PI / 2)
        got = [_exact_mc(name, lat, _key(seed) + d, k, X, beta) for d, (name, k) in enumerate(_batch_streams(case))]
        return {"mean": torch.stack([r[0] for r in got]), "var": torch.stack([r[1] for r in got])}
    name = case["diagram"]
    if kind == "energy":
        E, step = _energies(case, seed), _chunk(name, n, n_f)
        return {"values": torch.cat([_values(name, E[s:s + step], X, beta)[0] for s in range(0, n, step)], dim=1)}
    grads = kind in ("slope", "fused", "autograd")
    g = torch.from_numpy(_upstream(case, seed)).cuda() if grads else None
    mean, var, dX, params, values = _exact_mc(name, _lattice(name), _key(seed), n, X, beta, g, kind == "samples")
    if kind == "forward":
        return {"mean": mean, "var": var}
    if kind == "samples":
        return {"mean": mean, "var": var, "values": values}
    along = (g.conj() * dX).real
    if kind == "autograd":
        return {"sigma": mean, "g_omega": along, "g_mu": params[0], "g_kext": params[1:3]}
    return {"mean": mean, "var": var, "dSigma_dX": dX, "grad_X_re": along, "grad_params": params}

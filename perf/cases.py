"""The calls whose speed is measured: what a program does with this library,
from the smallest product to whole solves and whole DMRG runs.

Every case goes through the public entry points of ``binding``: products in
the three precisions that programs choose (float64, double-float, split
BF16), the product with its reverse mode under autograd, ground-state solves
(float64; mixed with refinement and the Hellmann-Feynman gradient), Lanczos
coefficients with their continued fraction, the device DMRG driver, and the
batched eigensolver of its truncation.

The operator blocks of a case come from its sizes (a model is the same model
on every call); couplings, wavefunctions, cotangents and density matrices
come from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_0902_3185_gb300 import binding
from workloads import lattice_models
from workloads.grown import grown_hubbard_superblock
from workloads.superblock import Superblock
from workloads.synthetic import random_sectored

# geometry, sites, electrons per spin, cut: the lattices of the tests and the benchmark
LATTICES = {
    "ladder12": ("ladder", 12, 5, 6),     # small 2-leg ladder, the smoke run's superblock
    "chain16": ("chain", 16, 8, None),
    "chain32": ("chain", 32, 16, None),   # half-filled Hubbard chain
    "ladder64": ("ladder", 64, 28, 33),   # 2 x 32 ladder at 1/8 hole doping
}


def listed():
    return [
        # one product on a small superblock: a user's own eigensolver or time
        # evolution on a short lattice, where launches and latency count
        dict(name="product_fp64_ladder12_m60", kind="product", blocks="ladder12", m=60, batch=2, prec="fp64"),
        # float64 product with wide ragged sectors (16..512)
        dict(name="product_fp64_sectors16", kind="product", blocks="random", sectors=16, dmin=16, dmax=512, batch=1,
             prec="fp64"),
        # the synthetic batched-matvec workload in split BF16: 64 sectors, 760 pairs
        dict(name="product_bf16x3_sectors64", kind="product", blocks="random", sectors=64, dmin=16, dmax=512, batch=1,
             prec="bf16x3"),
        # residual product with every term's expectation value, a sweep of 16
        # couplings on the m = 1000 ladder: observables and gradients of given states
        dict(name="term_dots_df64_ladder64_m1000", kind="term_dots", blocks="ladder64", m=1000, batch=16,
             prec="df64"),
        # forward and backward through autograd: fitting couplings to a target
        dict(name="autograd_fp64_chain32_m200", kind="autograd", blocks="chain32", m=200, batch=4, prec="fp64"),
        # float64 ground state of one superblock of a chain run at m = 200
        dict(name="ground_fp64_chain32_m200", kind="ground", blocks="chain32", m=200, batch=1, prec="fp64",
             grad=False),
        # one large superblock, as a DMRG step solves it: mixed, refined
        dict(name="ground_bf16x3_chain32_m1000", kind="ground", blocks="chain32", m=1000, batch=1, prec="bf16x3",
             grad=False),
        # a coupling sweep of 16 members on the m = 1000 ladder with gradients
        dict(name="ground_bf16x3_ladder64_m1000", kind="ground", blocks="ladder64", m=1000, batch=16, prec="bf16x3",
             grad=True),
        # local density of states: 100 Lanczos coefficients, 2001 frequencies
        dict(name="ldos_fp64_ladder64_m400", kind="ldos", blocks="ladder64", m=400, batch=4, coefs=100, points=2001),
        # a whole small DMRG run: Heisenberg chain, infinite algorithm and a sweep
        dict(name="dmrg_heisenberg16_m32", kind="dmrg", model="heisenberg", L=16, m=32, sweeps=1),
        # a whole DMRG run with larger blocks: Hubbard chain, infinite algorithm
        dict(name="dmrg_hubbard14_m160", kind="dmrg", model="hubbard_chain", L=14, m=160, sweeps=0),
        # density matrices of one truncation at m of about 1000: 12 sectors up to 300 wide
        dict(name="eig_sectors12_n300", kind="eig", sectors=12, n=300),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "term_dots", "autograd", "ground", "ground", "ldos", "dmrg", "eig"])
    if kind == "dmrg":
        model = rng.choice(["heisenberg", "j1j2", "hubbard_chain", "hubbard_ladder"])
        spin = model in ("heisenberg", "j1j2")
        return dict(kind=kind, model=model, L=rng.choice([10, 12, 14, 16] if spin else [6, 8, 10]),
                    m=_log_int(rng, 16, 64), sweeps=rng.choice([0, 1]))
    if kind == "eig":
        return dict(kind=kind, sectors=rng.randint(1, 12), n=_log_int(rng, 8, 300))
    if kind in ("product", "term_dots", "autograd") and rng.random() < 0.5:
        case = dict(kind=kind, blocks="random", sectors=rng.randint(3, 16), dmin=rng.randint(1, 16),
                    dmax=_log_int(rng, 20, 512), batch=rng.randint(1, 3))
        if kind != "product":
            case["dmax"] = min(case["dmax"], 200)
    else:
        blocks = rng.choice(sorted(LATTICES))
        top = {"ladder12": 150, "chain16": 200, "chain32": 400, "ladder64": 500}[blocks]
        case = dict(kind=kind, blocks=blocks, m=_log_int(rng, 30, top), batch=rng.randint(1, 8))
    if kind == "product":
        case["prec"] = rng.choice(["fp64", "df64", "bf16x3"])
    elif kind == "term_dots":
        case["prec"] = rng.choice(["fp64", "df64"])
    elif kind == "autograd":
        case["prec"] = "fp64"
    elif kind == "ground":
        case["prec"] = rng.choice(["fp64", "bf16x3"])
        case["grad"] = rng.random() < 0.5
        if case["prec"] == "fp64":
            case["m"], case["batch"] = min(case["m"], 250), min(case["batch"], 3)
    elif kind == "ldos":
        case["m"], case["batch"] = min(case["m"], 400), min(case["batch"], 4)
        case["coefs"], case["points"] = rng.randint(20, 100), rng.randint(200, 2001)
    return case


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=4)
def _blocks(blocks, m, sectors, dmin, dmax):
    """The operator blocks of a case: a model of these sizes, one batch member."""
    if blocks == "random":
        return random_sectored(seed=0, n_sectors=sectors, dmin=dmin, dmax=dmax)
    geometry, sites, n, cut = LATTICES[blocks]
    return grown_hubbard_superblock(sites, geometry, n, n, m=m, cut=cut, U_values=[8.0])


def _superblock(case, rng):
    sb = _blocks(case["blocks"], case.get("m"), case.get("sectors"), case.get("dmin"), case.get("dmax"))
    b = case["batch"]
    if case["blocks"] == "random":
        coeffs = 1.0 + 0.5 * rng.standard_normal((b, sb.n_terms))
        return sb.with_coeffs(coeffs)
    U = 4.0 + 8.0 * (np.arange(b) + rng.random(b)) / b  # one interaction per member
    couplings = np.stack([np.ones(b), U], axis=1)
    coeffs = sb.coeffs_from_couplings(couplings)
    return Superblock(sb.r, sb.c, coeffs, sb.pairs, sb.term_names, sb.class_names, sb.term_class, sb.term_mult,
                      couplings, sb.q_labels, dict(sb.meta))


def _normal(seed, shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _sizes(case):
    """Sector sizes of a truncation: largest in the middle, falling off to both sides."""
    k, n = case["sectors"], case["n"]
    mid, width = (k - 1) / 2, max(1.0, k / 3)
    return [max(1, int(round(n * math.exp(-0.5 * ((i - mid) / width) ** 2)))) for i in range(k)]


def _densities(case, seed):
    """Reduced density matrices (trace 1) of random sector blocks; their
    weights fall over two decades, as the kept states' of one sector do."""
    out = []
    for i, n in enumerate(_sizes(case)):
        q, r = torch.linalg.qr(_normal(seed * 64 + i, (n, n)))
        w = torch.logspace(0, -2, n, dtype=torch.float64, device="cuda") if n > 1 else torch.ones_like(q[0])
        rho = (q * w) @ q.T
        rho = rho + rho.T
        out.append(rho / rho.trace())
    return out


def _frequencies(points, batch, e0):
    w = torch.linspace(-20.0, 20.0, points, dtype=torch.float64, device="cuda")
    return torch.complex(e0 + w, torch.full_like(w, 0.1)).expand(batch, points).contiguous()


def _model(case, seed):
    rng = np.random.default_rng(seed)
    u = float(rng.random())
    name = case["model"]
    if name == "heisenberg":
        return lattice_models.heisenberg_chain(1.0 + 0.2 * u)
    if name == "j1j2":
        return lattice_models.heisenberg_chain(1.0, 0.1 + 0.3 * u)
    if name == "hubbard_chain":
        return lattice_models.hubbard_chain(1.0, 2.0 + 6.0 * u)
    return lattice_models.hubbard_ladder(1.0, 0.6 + 0.3 * u, 6.0)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case, seed=seed)
    if kind == "dmrg":
        s["desc"] = _model(case, seed)
        return s
    if kind == "eig":
        s["mats"] = _densities(case, seed)
        return s
    sb = _superblock(case, np.random.default_rng(seed))
    s["g"] = binding.GpuSuperblock(sb)
    s["x"] = _normal(seed, (sb.batch, sb.dim))
    if kind == "autograd":
        s["x"].requires_grad_(True)
        s["c"] = torch.tensor(sb.coeffs, device="cuda", requires_grad=True)
        s["cot"] = _normal(seed + (1 << 31), (sb.batch, sb.dim))
    if kind == "ldos":
        s["z"] = _frequencies(case["points"], sb.batch, 0.0)
    return s


# --------------------------------------------------------------------- run
def run(s):
    kind = s["kind"]
    if kind == "product":
        return s["g"].apply_H(s["x"], prec=s["prec"])
    if kind == "term_dots":
        y, dots = s["g"].apply_H_term_dots(s["x"], prec=s["prec"])
        return {"y": y, "dots": dots}
    if kind == "autograd":
        y = binding.apply_H(s["x"], s["c"], s["g"], s["prec"])
        dx, dc = torch.autograd.grad(y, (s["x"], s["c"]), s["cot"])
        return {"y": y.detach(), "dx": dx, "dc": dc}
    if kind == "ground":
        if s["prec"] == "fp64":
            out = s["g"].lanczos_ground(s["x"], tol=1e-12, max_iter=600, grad=s["grad"])
        else:  # the benchmark's mixed solve; a wavefunction good to nine digits asks for a tighter residual
            out = s["g"].lanczos_ground(s["x"], tol=2e-4, max_iter=300, prec=s["prec"], refine="newton_df64",
                                        refine_tol=1e-12, grad=s["grad"])
        if out[3] != 0:
            raise RuntimeError("the solve did not converge")
        res = {"e0": out[0], "psi": out[1]}
        if s["grad"]:
            res["dE"] = out[4]
        return res
    if kind == "ldos":
        norm2, a, b, n = s["g"].lanczos_coeffs(s["x"], s["coefs"])
        return {"norm2": norm2, "alpha": a, "beta": b, "n": n,
                "G": binding.continued_fraction(norm2, a, b, n, s["z"])}
    if kind == "dmrg":
        d = binding.GpuDmrg(s["desc"], s["L"], s["m"], guess=True)
        steps = d.infinite()
        if s["sweeps"]:
            steps += d.sweeps(s["sweeps"])
        d.close()
        return {k: np.array([st[k] for st in steps]) for k in ("energy", "eps_S", "eps_E")}
    out = []
    for w, v in binding.sym_eig_batched(s["mats"]):
        # an eigenvector has no sign of its own: the largest entry is made
        # positive, as programs do that store or compare them
        at = v.abs().argmax(dim=0, keepdim=True)
        out += [w, v * v.gather(0, at).sign()]
    return out


# -------------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass: operator blocks and vectors once, the
    multiply-adds of the cheaper order of every (term, sector pair) product;
    solves count the products and basis sweeps of their usual length."""
    kind = case["kind"]
    if kind == "eig":
        n = np.array(_sizes(case), dtype=np.float64)
        return {"bytes": float(8 * (2 * n * n + n).sum()), "flops": float((16 / 3 * n ** 3).sum())}
    if kind == "dmrg":
        d = 2 if case["model"] in ("heisenberg", "j1j2") else 4
        steps = case["L"] // 2 - 1 + case["sweeps"] * 2 * (case["L"] - 3)
        sectors = 6 if d == 2 else 20
        n = d * min(case["m"], d ** (case["L"] // 2 - 1)) / sectors  # a typical sector
        one = 30 * sectors * 4 * n ** 3 * (4 if d == 2 else 8) + 16 / 3 * sectors * n ** 3
        return {"bytes": float(steps * sectors * 8 * n * n * 8), "flops": float(steps * one)}
    sb = _superblock(case, np.random.default_rng(0))
    r, c, b = sb.r.astype(np.float64), sb.c.astype(np.float64), sb.batch
    flops, ops = 0.0, 0.0
    for p in sb.pairs:
        ro, ri, co, ci = r[p.s_out], r[p.s_in], c[p.s_out], c[p.s_in]
        if p.B is None:
            flops += 2 * ro * ri * co
        elif p.A is None:
            flops += 2 * ro * ci * co
        else:
            flops += min(2 * ro * ri * ci + 2 * ro * ci * co, 2 * ri * ci * co + 2 * ro * ri * co)
        ops += (0 if p.A is None else p.A.size) + (0 if p.B is None else p.B.size)
    flops *= b
    vec = 8.0 * b * sb.dim
    ops *= 8.0
    if kind == "product":
        return {"bytes": ops + 2 * vec, "flops": flops}
    if kind == "term_dots":
        return {"bytes": ops + 2 * vec, "flops": flops}
    if kind == "autograd":
        return {"bytes": ops + 4 * vec, "flops": 3 * flops}
    if kind == "ldos":
        j = case["coefs"]
        return {"bytes": j * (ops + vec) + j * j * vec, "flops": j * flops + 2.0 * j * j * sb.dim * b}
    j, extra = (150, 0) if case["prec"] == "fp64" else (60, 60)
    return {"bytes": j * (j * vec + ops + vec) + extra * (ops + 2 * vec),
            "flops": (j + extra) * flops + 2.0 * j * j * sb.dim * b}


# ------------------------------------------------------------------- exact
def _terms(sb, transpose=False):
    """Blocks of every pair on the device: (term, out slice, in slice, shapes, A, B)."""
    off = sb.offsets()
    out = []
    for p in sb.pairs:
        so, si = (p.s_in, p.s_out) if transpose else (p.s_out, p.s_in)
        if sb.r[so] * sb.c[so] == 0 or sb.r[si] * sb.c[si] == 0:
            continue
        A = None if p.A is None else torch.from_numpy(p.A).cuda()
        B = None if p.B is None else torch.from_numpy(p.B).cuda()
        if transpose:
            A, B = None if A is None else A.T.contiguous(), None if B is None else B.T.contiguous()
        out.append((p.term, slice(off[so], off[so + 1]), slice(off[si], off[si + 1]), (int(sb.r[si]), int(sb.c[si])),
                    A, B))
    return out


def _pair_product(x, t):
    _, _, src, (r, c), A, B = t
    z = x[:, src].reshape(-1, r, c)
    if B is not None:
        z = z @ B.T
    if A is not None:
        z = A @ z
    return z.reshape(x.shape[0], -1)


def _apply(terms, coeffs, x, y):
    y.zero_()
    for t in terms:
        y[:, t[1]] += coeffs[:, t[0], None] * _pair_product(x, t)
    return y


def _dots(terms, n_terms, x, g):
    d = torch.zeros(x.shape[0], n_terms, dtype=torch.float64, device="cuda")
    for t in terms:
        d[:, t[0]] += (g[:, t[1]] * _pair_product(x, t)).sum(dim=1)
    return d


def _replayed(terms, coeffs, shape):
    """The product captured once, replayed for every Lanczos step."""
    x = torch.zeros(shape, dtype=torch.float64, device="cuda")
    y = torch.zeros_like(x)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        _apply(terms, coeffs, x, y)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _apply(terms, coeffs, x, y)

    def product(v):
        x.copy_(v)
        graph.replay()
        return y.clone()

    return product


def _lanczos(product, x, n):
    """n Lanczos steps, every vector orthogonalised twice against all earlier ones."""
    v = x / x.norm(dim=1, keepdim=True)
    V = torch.empty(x.shape[0], n + 1, x.shape[1], dtype=torch.float64, device="cuda")
    a = torch.zeros(x.shape[0], n, dtype=torch.float64, device="cuda")
    b = torch.zeros_like(a)
    V[:, 0] = v
    for j in range(n):
        w = product(v)
        a[:, j] = (w * v).sum(dim=1)
        for _ in range(2):
            w = w - torch.bmm(torch.bmm(V[:, :j + 1], w[:, :, None]).transpose(1, 2), V[:, :j + 1])[:, 0]
        b[:, j] = w.norm(dim=1)
        v = w / b[:, j, None]
        V[:, j + 1] = v
    return a, b, V


def _ground(product, x, n=150, restarts=8):
    v = x
    for _ in range(restarts):
        a, b, V = _lanczos(product, v, n)
        T = torch.diag_embed(a) + torch.diag_embed(b[:, :-1], 1) + torch.diag_embed(b[:, :-1], -1)
        w, S = np.linalg.eigh(T.cpu().numpy())
        s = torch.from_numpy(np.ascontiguousarray(S[:, :, 0])).cuda()
        v = torch.bmm(s[:, None, :], V[:, :n])[:, 0]
        v = v / v.norm(dim=1, keepdim=True)
        hv = product(v)
        e0 = (v * hv).sum(dim=1)
        if float(((hv - e0[:, None] * v).norm(dim=1) / e0.abs().clamp(min=1.0)).max()) < 1e-14:
            break
    return e0, v * (v * x).sum(dim=1, keepdim=True).sign()


def exact(case, seed):
    kind = case["kind"]
    if kind == "dmrg":
        return None  # the energies of a truncated basis have no closed form
    if kind == "eig":
        out = []
        for rho in _densities(case, seed):
            w, v = torch.linalg.eigh(rho)
            w, v = w.flip(0), v.flip(1)
            out += [w, v * v.gather(0, v.abs().argmax(dim=0, keepdim=True)).sign()]
        return out
    sb = _superblock(case, np.random.default_rng(seed))
    terms = _terms(sb)
    coeffs = torch.from_numpy(sb.coeffs).cuda()
    x = _normal(seed, (sb.batch, sb.dim))
    y = torch.empty_like(x)
    if kind == "product":
        return _apply(terms, coeffs, x, y)
    if kind == "term_dots":
        return {"y": _apply(terms, coeffs, x, y), "dots": _dots(terms, sb.n_terms, x, x)}
    if kind == "autograd":
        cot = _normal(seed + (1 << 31), (sb.batch, sb.dim))
        return {"y": _apply(terms, coeffs, x, y),
                "dx": _apply(_terms(sb, transpose=True), coeffs, cot, torch.empty_like(x)),
                "dc": _dots(terms, sb.n_terms, x, cot)}
    product = _replayed(terms, coeffs, x.shape)
    if kind == "ground":
        e0, psi = _ground(product, x)
        res = {"e0": e0, "psi": psi}
        if case["grad"]:
            res["dE"] = _dots(terms, sb.n_terms, psi, psi)
        return res
    a, b, _ = _lanczos(product, x, case["coefs"])
    norm2 = (x * x).sum(dim=1)
    z = _frequencies(case["points"], sb.batch, 0.0)
    t = z - a[:, -1:]
    for j in range(case["coefs"] - 2, -1, -1):
        t = z - a[:, j:j + 1] - b[:, j:j + 1] ** 2 / t
    return {"norm2": norm2, "alpha": a, "beta": b, "n": None, "G": norm2[:, None] / t}

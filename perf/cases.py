"""The work whose speed this repository answers for, as calls a user's program makes.

Every case is a binary-glass spring network (glassgen's recipe, the only input family the tests, the
benchmark and the configurations use) and one pass through a public entry point on it:

  filter    Y = p_m(Ht) X on device blocks (pfe_filter_apply), the operator that everything else applies;
            FP64 or FP32, on the spring network's blocks or on general 3x3 blocks (a network under tension)
  adjoint   a training step on device buffers: the filter, its adjoint, the chain rule to springs and masses
  autograd  the same through torch.autograd from spring constants and masses (cheb_filter)
  solve     every eigenpair of an interval: filtered subspace iteration in FP64 or mixed precision, or
            block Lanczos
  batch     the same interval for several independent glasses in one call (pfe_solve_batch)

Large glasses are periodic supercells of a smaller one with their own spring constants per bond, so that
making inputs stays quick; the neighbour statistics are the generator's.
"""
import functools
import math
import weakref

import numpy as np
import torch

import glassgen
import paper_1902_07041_gb300 as pfe
from paper_1902_07041_gb300.autograd import SpringNetwork, cheb_filter


def listed():
    return [
        # the smallest useful call: a test-sized glass, few columns; launches and host work count
        dict(name="filter_small", kind="filter", atoms=1000, cells=1, k=16, m=40, dtype="f64", blocks="springs"),
        # odd sizes throughout: a ragged last column chunk and an odd number of steps
        dict(name="filter_ragged", kind="filter", atoms=5003, cells=1, k=33, m=101, dtype="f64", blocks="springs"),
        # one operator application of block Lanczos on the benchmark-sized glass (64 columns, degree 317)
        dict(name="filter_block", kind="filter", atoms=3700, cells=3, k=64, m=317, dtype="f64", blocks="springs"),
        # the subspace iteration's block on the benchmark-sized glass (994 columns), a short filter
        dict(name="filter_wide", kind="filter", atoms=3700, cells=3, k=994, m=24, dtype="f64", blocks="springs"),
        # a Hessian with transverse terms (a network under tension): full 3x3 blocks
        dict(name="filter_general", kind="filter", atoms=2500, cells=2, k=64, m=100, dtype="f64", blocks="tension"),
        # the FP32 filter of the mixed-precision modes on the benchmark-sized glass
        dict(name="filter_f32", kind="filter", atoms=3700, cells=3, k=128, m=200, dtype="f32", blocks="springs"),
        # gradients of a filtered block to X, springs and masses on device buffers
        dict(name="adjoint", kind="adjoint", atoms=2500, cells=2, k=32, m=60),
        # the same through torch.autograd, assembly of the Hessian included
        dict(name="autograd", kind="autograd", atoms=3001, cells=1, k=8, m=32),
        # all eigenpairs of the interval of the small configurations, FP64 subspace iteration (defaults)
        dict(name="solve_fp64", kind="solve", atoms=4000, cells=1, lo=0.02, hi=0.03, method=0, precision=0),
        # the batch configuration's interval on one of its sizes, defect-corrected FP32 filter
        dict(name="solve_mixed", kind="solve", atoms=1250, cells=2, lo=0.02, hi=0.026, method=0, precision=2),
        # block Lanczos, the production solver
        dict(name="solve_lanczos", kind="solve", atoms=4000, cells=1, lo=0.02, hi=0.03, method=1, precision=0),
        # several small samples in one call
        dict(name="solve_batch", kind="batch", atoms=700, samples=6, lo=0.02, hi=0.03),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _supercell(n):
    """(atoms, cells) of a glass of about n atoms whose generated cell stays small."""
    cells = 1 if n < 8000 else 2 if n < 48000 else 3
    return max(60, n // cells**3), cells


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "filter", "filter", "adjoint", "autograd", "solve", "batch"])
    if kind == "filter":
        atoms, cells = _supercell(_log(rng, 300, 100000))
        dtype, blocks = rng.choice([("f64", "springs")] * 3 + [("f32", "springs"), ("f64", "tension")])
        k, m = _log(rng, 1, 1000), _log(rng, 8, 700)
        most = 1.1e9  # atoms x columns x steps, about half of the largest listed filter
        m = max(8, min(m, int(most / (atoms * cells**3 * k))))
        k = max(1, min(k, int(most / (atoms * cells**3 * m))))
        return dict(kind=kind, atoms=atoms, cells=cells, k=k, m=m, dtype=dtype, blocks=blocks)
    if kind == "adjoint":
        atoms, cells = _supercell(_log(rng, 300, 20000))
        return dict(kind=kind, atoms=atoms, cells=cells, k=_log(rng, 1, 40), m=_log(rng, 5, 70))
    if kind == "autograd":
        return dict(kind=kind, atoms=_log(rng, 200, 6000), cells=1, k=_log(rng, 1, 32), m=_log(rng, 5, 60))
    lo = round(rng.uniform(0.015, 0.03), 4)
    if kind == "solve":
        method, precision = rng.choice([(0, 0), (0, 2), (1, 0)])
        return dict(kind=kind, atoms=_log(rng, 800, 4000), cells=1, lo=lo, hi=round(lo + rng.uniform(0.005, 0.01), 4),
                    method=method, precision=precision)
    return dict(kind=kind, atoms=_log(rng, 300, 1000), samples=rng.randint(2, 8), lo=lo,
                hi=round(lo + rng.uniform(0.005, 0.01), 4))


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=16)
def _glass(atoms):
    return glassgen.generate(atoms, 17)


class Network:
    """A spring network: bonds (bi, bj), unit vectors, spring constants, masses (host arrays).  The positions
    follow from the size, the spring constants and the species on the sites from the seed."""

    def __init__(self, atoms, cells, seed):
        g = _glass(atoms)
        self.n_atoms = atoms * cells**3
        # bond (i, j) of the cell joins image a of atom i with image a + shift of atom j
        shift = -np.rint((g.pos[g.bj] - g.pos[g.bi]) / g.box).astype(np.int64)
        a = np.stack(np.meshgrid(*[np.arange(cells)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
        b = (a + shift[None]) % cells
        flat = np.array([cells * cells, cells, 1])
        bi = ((a @ flat) * atoms + g.bi[None]).reshape(-1)
        bj = ((b @ flat) * atoms + g.bj[None]).reshape(-1)
        self.bi, self.bj = bi.astype(np.int32), bj.astype(np.int32)
        self.rhat = np.tile(g.rhat, (cells**3, 1))
        rng = np.random.default_rng(seed)
        self.k = glassgen.K_MEDIAN * np.exp(glassgen.K_SIGMA * rng.standard_normal(bi.size))
        self.mass = rng.permutation(np.tile(g.mass, cells**3))


def _operator(net, tension=0.0, device="cuda"):
    """x -> H x on (3N, k) FP64 tensors, from the bonds: H = M^-1/2 Delta M^-1/2 with
    Delta_ij = -(k r r^T + tension k (I - r r^T)); differentiable in springs and masses."""
    bi = torch.from_numpy(np.ascontiguousarray(net.bi, np.int64)).to(device)
    bj = torch.from_numpy(np.ascontiguousarray(net.bj, np.int64)).to(device)
    r = torch.from_numpy(np.ascontiguousarray(net.rhat)).to(device).unsqueeze(-1)

    def apply(x, springs, masses):
        x = x.reshape(net.n_atoms, 3, -1)
        w = masses.rsqrt().reshape(-1, 1, 1)
        y = x * w
        delta = y.index_select(0, bi) - y.index_select(0, bj)
        f = r * (r * delta).sum(1, keepdim=True)
        if tension:
            f = (1.0 - tension) * f + tension * delta
        f = f * springs.reshape(-1, 1, 1)
        out = torch.zeros_like(y).index_add(0, bi, f).index_add(0, bj, f, alpha=-1.0)
        return (out * w).reshape(3 * net.n_atoms, -1)

    return apply


def _springs(net, device="cuda"):
    return torch.from_numpy(net.k).to(device), torch.from_numpy(net.mass).to(device)


def _lambda_max(net, tension=0.0):
    """An upper bound of the spectrum as a user may know it: 5 % above a power iteration's value."""
    apply, (ks, ms) = _operator(net, tension), _springs(net)
    x = torch.randn(3 * net.n_atoms, 1, dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(1))
    for _ in range(60):
        x = apply(x / x.norm(), ks, ms)
    return float("%.3g" % (1.05 * float(x.norm())))


def _coefficients(m, xi=-0.96, eta=-0.94):
    """Chebyshev series of the indicator of [xi, eta] with Lanczos sigma damping."""
    j = np.arange(1, m + 1)
    a, b = math.acos(xi), math.acos(eta)
    c = np.empty(m + 1)
    c[0] = (a - b) / math.pi
    c[1:] = 2.0 / (math.pi * j) * (np.sin(j * a) - np.sin(j * b)) * np.sinc(j / (m + 1.0))
    return c


def _tension(case):
    return 0.05 if case.get("blocks") == "tension" else 0.0


def _bsr(net, tension):
    """Delta as 3x3 block CSR with ascending columns, for a network under tension."""
    n = net.n_atoms
    rr = net.rhat[:, :, None] * net.rhat[:, None, :]
    blk = net.k[:, None, None] * (rr + tension * (np.eye(3) - rr))
    diag = np.zeros((n, 3, 3))
    np.add.at(diag, net.bi, blk)
    np.add.at(diag, net.bj, blk)
    row = np.concatenate([net.bi, net.bj, np.arange(n)])
    col = np.concatenate([net.bj, net.bi, np.arange(n)])
    order = np.lexsort((col, row))
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(row, minlength=n), out=rp[1:])
    return rp, col[order].astype(np.int32), np.concatenate([-blk, -blk, diag])[order].reshape(-1)


class State:
    """What the user's program holds; the contexts are released with it."""

    def __init__(self, case, **held):
        self.case = case
        self.__dict__.update(held)
        for c in self.ctxs:
            weakref.finalize(self, pfe.pfe_destroy, c)


def _context(net, tension=0.0):
    if tension:
        rp, ci, vals = _bsr(net, tension)
    else:
        rp, ci, vals = pfe.pfe_springs_to_bsr(net.n_atoms, net.bi, net.bj, net.k, net.rhat)
    return pfe.pfe_create(net.n_atoms, rp, ci, vals, net.mass), ci.size


def _block(case, net, seed, which=0):
    """A column-major n x k block of normals, as (k, n) storage."""
    g = torch.Generator("cuda").manual_seed(2 * seed + which)
    return torch.randn(case["k"], 3 * net.n_atoms, dtype=torch.float64, device="cuda", generator=g)


def _networks(case, seed):
    if case["kind"] != "batch":
        return [Network(case["atoms"], case["cells"], seed)]
    return [Network(case["atoms"] + 37 * i, 1, seed + 101 * i) for i in range(case["samples"])]


def prepare(case, seed):
    nets = _networks(case, seed)
    net, kind = nets[0], case["kind"]
    if kind == "autograd":
        ks, ms = _springs(net)
        return State(case, ctxs=[], net=SpringNetwork(net.n_atoms, net.bi, net.bj, net.rhat), lmax=_lambda_max(net),
                     X=_block(case, net, seed).t().contiguous().requires_grad_(), ks=ks.requires_grad_(),
                     ms=ms.requires_grad_(), Ybar=_block(case, net, seed, 1).t().contiguous(), coef=_coefficients(case["m"]))
    if kind in ("solve", "batch"):
        ctxs = []
        for t in nets:
            ctx, _ = _context(t)
            lmax = _lambda_max(t)
            pfe.pfe_set_interval(ctx, case["lo"] * lmax, case["hi"] * lmax)
            pfe.pfe_set_param(ctx, pfe.PFE_P_METHOD, case.get("method", 0))
            pfe.pfe_set_param(ctx, pfe.PFE_P_PRECISION, case.get("precision", 0))
            ctxs.append(ctx)
        return State(case, ctxs=ctxs, n=[3 * t.n_atoms for t in nets],
                     field=[_field(3 * t.n_atoms, seed) for t in nets])
    ctx, nnzb = _context(net, _tension(case))
    pfe.pfe_set_param(ctx, pfe.PFE_P_LAMBDA_MAX, _lambda_max(net, _tension(case)))
    X = _block(case, net, seed)
    if kind == "filter":
        X = X.to(torch.float32) if case["dtype"] == "f32" else X
        return State(case, ctxs=[ctx], n=3 * net.n_atoms, X=X, Y=torch.empty_like(X), coef=_coefficients(case["m"]))
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (net.bi, net.bj, net.rhat)]
    return State(case, ctxs=[ctx], n=3 * net.n_atoms, X=X, Y=torch.empty_like(X), Ybar=_block(case, net, seed, 1),
                 Xbar=torch.empty_like(X), bonds=dev, coef=_coefficients(case["m"]),
                 vbar=torch.empty(9 * nnzb, dtype=torch.float64, device="cuda"),
                 kbar=torch.empty(net.k.size, dtype=torch.float64, device="cuda"),
                 mbar=torch.empty(net.n_atoms, dtype=torch.float64, device="cuda"))


def _capacity(n, case):
    """Room for the eigenpairs of the interval, about twice the measured density (5 per 1,000 atoms and 0.001)."""
    return int(10.0 * n / 3000 * (case["hi"] - case["lo"]) / 0.001) + 32


def _field(n, seed):
    """Four displacement fields to project onto the modes of the interval."""
    return torch.randn(n, 4, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed + 5))


# ---------------------------------------------------------------- one pass
def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "filter":
        pfe.pfe_filter_apply(s.ctxs[0], case["m"], s.coef, case["k"], s.X, s.n, s.Y, s.n,
                             pfe.PFE_F32 if case["dtype"] == "f32" else pfe.PFE_F64)
        return s.Y
    if kind == "adjoint":
        ctx, m, k, n = s.ctxs[0], case["m"], case["k"], s.n
        pfe.pfe_filter_apply(ctx, m, s.coef, k, s.X, n, s.Y, n, pfe.PFE_F64)
        pfe.pfe_filter_adjoint(ctx, m, s.coef, k, s.X, n, s.Ybar, n, s.Xbar, n, s.vbar)
        pfe.pfe_chain_springs(ctx, s.kbar.numel(), *s.bonds, s.vbar, s.kbar, s.mbar)
        return {"Y": s.Y, "Xbar": s.Xbar, "vals_bar": s.vbar, "k_bar": s.kbar, "m_bar": s.mbar}
    if kind == "autograd":
        Y = cheb_filter(s.X, s.ks, s.ms, s.net, s.coef, s.lmax)
        gx, gk, gm = torch.autograd.grad(Y, (s.X, s.ks, s.ms), s.Ybar)
        return {"Y": Y.detach(), "X": gx, "k": gk, "m": gm}
    if kind == "solve":
        found = [pfe.pfe_solve(s.ctxs[0])[0]]
    else:
        found, status = pfe.pfe_solve_batch(s.ctxs)
        if status != pfe.PFE_OK:
            raise RuntimeError("pfe_solve_batch: status %d" % status)
    # Eigenvectors are defined up to sign (and rotation among close ones): what a program uses and what can be
    # compared is their action, here the part of given fields inside the interval.  With the FP32 filter they
    # are determined only to TOL / gap, so that case gives its eigenvalues.
    lams, parts = [], []
    for ctx, n, nf, f in zip(s.ctxs, s.n, found, s.field):
        cap = _capacity(n, case)
        V = torch.empty(cap, n, dtype=torch.float64, device="cuda")
        lams.append(pfe.pfe_get_eigenpairs(ctx, n, cap, vecs_out=V)[0])
        V = V[:nf]
        parts.append(V.t() @ (V @ f))
    if case.get("precision", 0):
        return {"lambda": lams}
    return {"lambda": lams, "part": parts}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    n_atoms = case["atoms"] * case.get("cells", 1) ** 3
    kind = case["kind"]
    noff = 10.28 * n_atoms  # off-diagonal blocks of the recipe (both directions)
    full = _tension(case) > 0
    per_col = 18.0 * (noff + n_atoms) if full else 12.0 * noff + 18.0 * n_atoms  # one product with H
    per_col += 4.0 * 3 * n_atoms  # the recurrence and the sum
    es = 4 if case.get("dtype") == "f32" else 8
    matrix = noff * (9 if full else 3) * es + noff * 4 + 6 * n_atoms * es
    if kind == "filter":
        return {"bytes": 2 * 3 * n_atoms * case["k"] * es + matrix, "flops": per_col * case["k"] * case["m"]}
    if kind in ("adjoint", "autograd"):
        outer = 18.0 * (noff + n_atoms) * case["k"] * case["m"]
        return {"bytes": 4 * 3 * n_atoms * case["k"] * 8 + 2 * matrix + (noff + n_atoms) * 72,
                "flops": 3 * per_col * case["k"] * case["m"] + outer}
    if kind == "batch":
        n_atoms = sum(case["atoms"] + 37 * i for i in range(case["samples"]))
    # modes by the measured density (about 5 per 1,000 atoms and 0.001 of the spectrum near 0.025), width 1.5x,
    # six iterations of a filter whose degree follows the interval, and the dense steps of each
    modes = 5.0 * n_atoms / 1000 * (case["hi"] - case["lo"]) / 0.001
    q = 1.5 * modes / case.get("samples", 1) + 16
    m = 1.2 / (case["hi"] - case["lo"])
    per_atom = per_col / (case["atoms"] * case.get("cells", 1) ** 3)
    return {"bytes": 3 * n_atoms * modes / case.get("samples", 1) * 8 + 112 * 11.3 * n_atoms,
            "flops": 6 * (per_atom * n_atoms * q * m + 5.5 * 3 * n_atoms * q * q)}


# ---------------------------------------------------------------- the same in plain torch, 64 bits
def _chebyshev(apply, X, coef, lmax):
    c = d = 0.5 * lmax
    t0, t1 = X, (apply(X) - c * X) / d
    y = coef[0] * t0 + coef[1] * t1
    for g in coef[2:]:
        t0, t1 = t1, 2.0 * (apply(t1) - c * t1) / d - t0
        y = y + g * t1
    return y


def exact(case, seed):
    kind, nets = case["kind"], _networks(case, seed)
    net = nets[0]
    ks, ms = _springs(net)
    if kind in ("solve", "batch"):
        if net.n_atoms > 4200:  # a dense solver would take too long
            return None
        lams, parts = [], []
        for t in nets:
            lam, part = _eigen(t, case, seed)
            lams.append(lam)
            parts.append(part)
        return {"lambda": lams} if case.get("precision", 0) else {"lambda": lams, "part": parts}
    apply, lmax, coef = _operator(net, _tension(case)), _lambda_max(net, _tension(case)), _coefficients(case["m"])
    X = _block(case, net, seed)
    if kind == "filter":
        Y = torch.empty_like(X)
        X = X.to(torch.float32).double() if case["dtype"] == "f32" else X
        for c in range(0, case["k"], 128):  # the bond sums of all columns at once would not fit
            Y[c:c + 128] = _chebyshev(lambda x: apply(x, ks, ms), X[c:c + 128].t().contiguous(), coef, lmax).t()
        return Y
    X = X.t().contiguous().requires_grad_()
    ks.requires_grad_()
    ms.requires_grad_()
    Y = _chebyshev(lambda x: apply(x, ks, ms), X, coef, lmax)
    Ybar = _block(case, net, seed, 1)
    gx, gk, gm = torch.autograd.grad(Y, (X, ks, ms), Ybar.t())
    if kind == "adjoint":
        return {"Y": Y.detach().t(), "Xbar": gx.t(), "vals_bar": None, "k_bar": gk, "m_bar": gm}
    return {"Y": Y.detach(), "X": gx, "k": gk, "m": gm}


def _eigen(net, case, seed):
    """Eigenvalues in the interval and the fields' parts, by a dense solver; the vectors only for small glasses
    (for large ones they would take too long)."""
    n = 3 * net.n_atoms
    apply, (ks, ms), lmax = _operator(net), _springs(net), _lambda_max(net)
    H = torch.empty(n, n, dtype=torch.float64, device="cuda")
    for c in range(0, n, 512):
        e = torch.zeros(n, min(512, n - c), dtype=torch.float64, device="cuda")
        e[torch.arange(c, c + e.shape[1]), torch.arange(e.shape[1])] = 1.0
        H[:, c:c + e.shape[1]] = apply(e, ks, ms)
    H = 0.5 * (H + H.t())
    lo, hi = case["lo"] * lmax, case["hi"] * lmax
    if net.n_atoms > 1500:
        w = torch.linalg.eigvalsh(H)
        return _padded(w[(w >= lo) & (w <= hi)], n, case), None
    w, V = torch.linalg.eigh(H)
    at = (w >= lo) & (w <= hi)
    V = V[:, at]
    return _padded(w[at], n, case), V @ (V.t() @ _field(n, seed))


def _padded(w, n, case):
    out = np.zeros(_capacity(n, case))
    out[:w.numel()] = w.cpu().numpy()
    return out

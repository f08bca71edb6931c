"""The measured workloads: the work a user of the package has it do, through the public ``Context`` calls.

Sizes are the named molecule shapes of the repository (tiny o=4 v=8, CO o=14 v=42, butadiene o=30 v=130,
benzene o=42 v=186) and ragged ones between them. Inputs follow the repository's recipe (orbital energies
uniform in two bands, a random real integral tensor with the 8-fold permutational symmetry, MP2-like
doubles, Lambda = T), generated on the GPU from the seed alone. Solves run to residuals near the floor of
the FP64-accurate residual, so that their results do not carry the rounding of the inner arithmetic. The
low-precision sigma is measured inside the solves that use it (it has no other use than as their inner
operator).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1902_06016_gb300 import Context

WINDOW = (-1.0, -0.2)      # ionisation window [Ha]
EA_WINDOW = (0.1, 0.9)     # attachment window [Ha]
LU_MAX = 6000              # largest dimension whose dense solves give the exact values in seconds


# ---- the cases --------------------------------------------------------------------------------------
def listed():
    return [
        # smallest call: the operator applied to one block of vectors (an outer program's own iteration)
        dict(name="sigma_fp64_tiny", kind="sigma", o=4, v=8, nvec=12, precision="fp64", transpose=False),
        # the full spectrum of a model system in plain FP64: all spin-orbitals on a 200-point grid
        dict(name="solve_fp64_tiny", kind="solve", sector="ip", o=4, v=8, norb=12, nw=200, eta=0.01,
             precision="fp64", tol=1e-11, vectors=False),
        # reference-quality G of a small molecule: FP64-accurate inner operator, every spin-orbital
        dict(name="solve_exact_co", kind="solve", sector="ip", o=14, v=42, norb=56, nw=10, eta=0.01,
             precision="fp64_tc", tol=1e-10, vectors=False),
        # the other half of G (electron attachment), ragged size
        dict(name="solve_tf32_ea", kind="solve", sector="ea", o=9, v=33, norb=33, nw=8, eta=0.05,
             precision="tf32", tol=1e-10, vectors=False),
        # bf16 inner operator, ragged size, solution vectors kept
        dict(name="solve_bf16_odd", kind="solve", sector="ip", o=23, v=77, norb=23, nw=9, eta=0.01,
             precision="bf16", tol=1e-10, vectors=True),
        # full-dimension solves of the occupied block of a mid-sized molecule
        dict(name="solve_tf32_butadiene", kind="solve", sector="ip", o=30, v=130, norb=30, nw=12, eta=0.005,
             precision="tf32", tol=1e-10, vectors=False),
        # one FP64-accurate operator application (residuals, Krylov models) at the largest molecule
        dict(name="sigma_exact_benzene", kind="sigma", o=42, v=186, nvec=84, precision="fp64_tc", transpose=False),
        # a new molecule: the similarity-transformed operator is built and applied for the first time
        dict(name="init_benzene", kind="init", o=42, v=186, nvec=2, precision="tf32"),
        # the spectrum on a dense grid from a reduced model in hand (order 336)
        dict(name="eval_benzene", kind="eval", o=42, v=186, norb=42, seeds=8, nw=2000, eta=0.01, tol=1e-10),
        # the same for all 160 spin-orbitals of butadiene (order 800)
        dict(name="eval_large_order", kind="eval", o=30, v=130, norb=160, seeds=5, nw=240, eta=0.01, tol=1e-10),
        # a backward pass: G and the gradient with respect to the doubles (forward and adjoint solves)
        dict(name="gradient_odd", kind="gradient", o=19, v=67, norb=19, nw=5, eta=0.03, precision="tf32", tol=1e-10),
        # the whole method on a new molecule: operator, reduced model, refinement, spectrum
        dict(name="spectrum_butadiene", kind="spectrum", o=30, v=130, norb=30, seeds=8, nw=1000, eta=0.01, tol=1e-10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (costs bounded by the listed ones of its kind)."""
    kind = rng.choice(["sigma", "sigma", "solve", "solve", "solve", "init", "eval", "eval", "gradient", "spectrum"])
    if kind == "sigma":
        prec = rng.choice(["fp64", "fp64_tc", "fp64_tc"])
        o = _log(rng, 4, 14 if prec == "fp64" else 42)
        v = _log(rng, max(5, 2 * o), max(12, int(4.4 * o)))
        return dict(kind=kind, o=o, v=v, nvec=_log(rng, 1, 84), precision=prec, transpose=rng.random() < 0.3)
    if kind == "solve":
        prec = rng.choice(["fp64", "fp64_tc", "tf32", "tf32", "bf16"])
        sector = rng.choice(["ip", "ip", "ip", "ea"])
        if sector == "ea":
            o = _log(rng, 3, 9)
            v = _log(rng, 2 * o, int(3.6 * o))
        else:
            o = _log(rng, 4, 6 if prec == "fp64" else 14 if prec == "fp64_tc" else 30)
            v = _log(rng, 2 * o, int(4.3 * o))
        norb = rng.randint(1, v if sector == "ea" else o)
        return dict(kind=kind, sector=sector, o=o, v=v, norb=norb, nw=_log(rng, 1, 12),
                    eta=0.05 if sector == "ea" else rng.choice([0.01, 0.005]), precision=prec,
                    tol=1e-11 if prec == "fp64" else 1e-10, vectors=rng.random() < 0.3)
    if kind == "init":
        o = _log(rng, 4, 42)
        return dict(kind=kind, o=o, v=_log(rng, 2 * o, int(4.4 * o)), nvec=rng.randint(1, 4),
                    precision=rng.choice(["tf32", "bf16"]))
    if kind == "eval":
        o = _log(rng, 6, 30)
        v = _log(rng, 2 * o, int(4.3 * o))
        return dict(kind=kind, o=o, v=v, norb=rng.randint(2, o), seeds=rng.randint(2, 8), nw=_log(rng, 50, 2000),
                    eta=0.01, tol=1e-10)
    if kind == "gradient":
        o = _log(rng, 5, 21)
        return dict(kind=kind, o=o, v=_log(rng, 2 * o, int(3.5 * o)), norb=rng.randint(1, o), nw=rng.randint(1, 5),
                    eta=0.03, precision=rng.choice(["tf32", "bf16"]), tol=1e-10)
    o = _log(rng, 10, 28)
    return dict(kind=kind, o=o, v=_log(rng, 2 * o, int(4.3 * o)), norb=rng.randint(2, o), seeds=rng.randint(5, 8),
                nw=_log(rng, 100, 1000), eta=0.01, tol=1e-10)


# ---- inputs -----------------------------------------------------------------------------------------
def _i64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _lsr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _uniform(key, salt):
    """Uniform (0, 1) doubles, a pure function of (key, salt): the SplitMix64 output function."""
    z = (key + salt + 1) * _i64(0x9E3779B97F4A7C15)
    z = (z ^ _lsr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _lsr(z, 27)) * _i64(0x94D049BB133111EB)
    return (_lsr(z ^ _lsr(z, 31), 11).double() + 0.5) * 2.0 ** -53


def _normal(key, salt):
    u = _uniform(key * 2, salt)
    return torch.sqrt(-2.0 * torch.log(u)) * torch.cos(2.0 * math.pi * _uniform(key * 2 + 1, salt))


def _canon(p, q):
    hi, lo = torch.maximum(p, q), torch.minimum(p, q)
    return hi * (hi + 1) // 2 + lo


def _antisym(salt, scale, P, Q, R, S):
    """<pq||rs> = (pr|qs) - (ps|qr) for broadcastable index tensors."""
    direct = _normal(_canon(_canon(P, R), _canon(Q, S)), salt)
    return scale * (direct - _normal(_canon(_canon(P, S), _canon(Q, R)), salt))


def _pairs(k):
    """(first, second) index of every pair a < b in the packed order b (b - 1) / 2 + a."""
    b, a = torch.tril_indices(k, k, -1, device="cuda")
    return a, b


def _inputs(case, seed):
    o, v = case["o"], case["v"]
    salt = _i64((seed * 0x2545F4914F6CDD1D + 0x1234567) % (1 << 64))
    scale = 0.05 * math.sqrt(4.0 * 8.0 ** 2 / (o * v * v))   # keeps the correlation shift of the poles size-independent
    n = torch.arange(o + v, device="cuda")
    O, V = n[:o], n[o:]

    def block(P, Q, R, S):
        out = torch.empty((len(P), len(Q), len(R), len(S)), dtype=torch.float64, device="cuda")
        step = max(1, (1 << 26) // max(1, out[0].numel()))
        for i in range(0, len(P), step):
            out[i:i + step] = _antisym(salt, scale, P[i:i + step, None, None, None], Q[:, None, None], R[:, None], S)
        return out

    x = SimpleNamespace(o=o, v=v)
    eps_o = -1.5 + 1.2 * _uniform(n[:o] + (1 << 50), salt)
    eps_v = 0.1 + 1.9 * _uniform(n[o:] + (1 << 51), salt)
    x.eps = torch.cat([eps_o, eps_v])
    x.oooo, x.ooov, x.oovv = block(O, O, O, O), block(O, O, O, V), block(O, O, V, V)
    x.ovov, x.ovvv = block(O, V, O, V), block(O, V, V, V)
    x.t1 = 0.01 * _normal(torch.arange(o * v, device="cuda") + (1 << 52), salt).reshape(o, v)
    x.t2 = x.oovv / (eps_o[:, None, None, None] + eps_o[:, None, None] - eps_v[:, None] - eps_v)
    x.l1, x.l2 = x.t1.clone(), x.t2.clone()
    x.vvvv = None
    if case.get("sector") == "ea":
        a, b = _pairs(v)
        a, b = a + o, b + o
        x.vvvv = _antisym(salt, scale, a[:, None], b[:, None], a, b).contiguous()
    return x


def _dim(case):
    o, v = case["o"], case["v"]
    return v + v * (v - 1) // 2 * o if case.get("sector") == "ea" else o + o * (o - 1) // 2 * v


def _block(case, seed):
    """A block of complex vectors, one per row, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed * 7 + 3)
    return torch.randn(case["nvec"], _dim(case), dtype=torch.complex128, device="cuda", generator=g)


def _freqs(case, seed):
    """The output grid: uniform over the window, shifted by less than one spacing."""
    lo, hi = EA_WINDOW if case.get("sector") == "ea" else WINDOW
    n = case["nw"]
    shift = np.random.RandomState(seed % (1 << 31)).uniform(0.0, 1.0)
    return lo + (hi - lo) * (np.arange(n) + shift) / n


def _orbitals(case):
    o = case["o"]
    return list(range(o, o + case["norb"])) if case.get("sector") == "ea" else list(range(case["norb"]))


def _seeds(case):
    return np.linspace(*WINDOW, case["seeds"])


def _gbar(case, seed):
    r = np.random.RandomState((seed + 11) % (1 << 31))
    shape = (case["nw"], case["norb"], case["norb"])
    return r.standard_normal(shape) + 1j * r.standard_normal(shape)


def prepare(case, seed):
    s = SimpleNamespace(case=case)
    kind = case["kind"]
    inp = _inputs(case, seed)
    if kind in ("sigma", "init"):
        s.X = _block(case, seed)
        if kind == "init":
            s.inp = inp
            return s
        s.out = torch.empty_like(s.X)
        s.ctx = Context(inp)
        s.ctx.sigma(s.X[:1].clone(), precision=case["precision"], transpose=case["transpose"])   # operands laid out
        return s
    s.orb, s.w = _orbitals(case), _freqs(case, seed)
    if kind == "spectrum":
        s.inp = inp
    else:
        s.ctx = Context(inp, tol=case["tol"], precision=case.get("precision", "tf32"),
                        sector=case.get("sector", "ip"), vvvv=inp.vvvv)
    n = case["norb"]
    if kind == "solve" and case["vectors"]:
        s.X = torch.empty((len(s.w), n, s.ctx.D), dtype=torch.complex128, device="cuda")
    if kind == "gradient":
        s.gbar = _gbar(case, seed)
    if kind in ("eval", "spectrum"):
        s.G = torch.empty((len(s.w), n, n), dtype=torch.complex128, device="cuda")
        s.A = torch.empty(len(s.w), dtype=torch.float64, device="cuda")
    if kind == "eval":
        s.ctx.mor_build(_seeds(case), case["eta"], s.orb)
        s.ctx.mor_eval(s.w[:1], want_A=False)   # the model's Hessenberg form, kept by the context
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "sigma":
        return s.ctx.sigma(s.X, precision=c["precision"], transpose=c["transpose"], out=s.out)
    if kind == "init":
        ctx = Context(s.inp, precision=c["precision"])
        y = ctx.sigma(s.X, precision="fp64_tc")
        ctx.close()
        return y
    if kind == "solve":
        r = s.ctx.solve_full(s.w, c["eta"], s.orb, want_A=False, want_X=c["vectors"], X=s.X if c["vectors"] else None)
        return {"G": r["G"], "X": r["X"]}
    if kind == "gradient":
        G, g = s.ctx.green_grad_t2(s.w, c["eta"], s.orb, s.gbar)
        return {"G": G, "g": g}
    if kind == "eval":
        r = s.ctx.mor_eval(s.w, G=s.G, A=s.A)
        return {"G": r["G"], "A": r["A"]}
    ctx = Context(s.inp, tol=c["tol"], precision="tf32")
    ctx.mor_build(_seeds(c), c["eta"], s.orb)
    ctx.mor_refine(*WINDOW, 500, 1e-6, 1700)
    r = ctx.mor_eval(s.w, G=s.G, A=s.A)
    ctx.close()
    return {"G": r["G"], "A": r["A"]}


# ---- the work a pass cannot do without ----------------------------------------------------------------
def _operator(case):
    """(flops of one application to a complex vector, elements of the operator's blocks)"""
    o, v = case["o"], case["v"]
    if case.get("sector") == "ea":
        o, v = v, o                # the attachment operator has the ionisation one's blocks with o and v exchanged
    P = o * (o - 1) // 2
    flops = 2.0 * (2.0 * (o * v) ** 2 * o + 2.0 * P * P * v + 4.0 * P * v * v + 4.0 * o * P * v)
    return flops, float((o * v) ** 2 + P * P + 2 * P * v * (v + o) + o * o)


def _input_elements(case):
    o, v = case["o"], case["v"]
    return float(o ** 4 + o ** 3 * v + 3 * (o * v) ** 2 + (o * v) ** 2 + o * v ** 3 + 2 * o * v + o + v)


def _init_flops(case):
    """The three largest contractions of the operator build and the oooo one."""
    o, v = case["o"], case["v"]
    return 2.0 * (o * v) ** 3 + 2.0 * (o * v) * (o * o) * (v * v) + 2.0 * 2.0 * (o ** 4) * (v ** 2) + 2.0 * o * o * v ** 3 * o


def work(case):
    kind = case["kind"]
    f1, blocks = _operator(case)
    D = _dim(case)
    if kind == "sigma":
        return {"bytes": 8.0 * blocks + 32.0 * D * case["nvec"], "flops": f1 * case["nvec"]}
    if kind == "init":
        return {"bytes": 8.0 * _input_elements(case) + 8.0 * blocks + 32.0 * D * case["nvec"],
                "flops": _init_flops(case) + f1 * case["nvec"]}
    n, nw = case["norb"], case["nw"]
    g_bytes = 16.0 * nw * n * n
    if kind == "solve":   # at least one application per column, its right-hand side read and solution reduced
        x = 16.0 * D * n * nw if case["vectors"] else 0.0
        return {"bytes": 8.0 * blocks + 16.0 * D * n + g_bytes + x, "flops": f1 * n * nw}
    if kind == "gradient":   # forward and adjoint columns, and the contraction of both into the gradient
        return {"bytes": 8.0 * blocks + 16.0 * D * n + 2.0 * g_bytes + 8.0 * (case["o"] * case["v"]) ** 2,
                "flops": 3.0 * f1 * n * nw}
    m = n * case["seeds"]
    solve = 8.0 * nw * (0.5 * m * m * n + m * n * n)    # back substitution and the contraction with the left vectors
    if kind == "eval":
        return {"bytes": 16.0 * (m * m + 2.0 * m * n) + g_bytes, "flops": solve}
    return {"bytes": 8.0 * _input_elements(case) + 8.0 * blocks + 32.0 * D * m + g_bytes,
            "flops": _init_flops(case) + f1 * m + solve}


# ---- the same in 64 bits by plain torch ----------------------------------------------------------------
E = torch.einsum


def _common(x):
    """Elements of the similarity-transformed Hamiltonian that both halves share."""
    o = x.o
    h = SimpleNamespace()
    h.tau = x.t2 + E("ia,jb->ijab", x.t1, x.t1) - E("ib,ja->ijab", x.t1, x.t1)
    h.Fme = E("nf,mnef->me", x.t1, x.oovv)
    h.Fmi = torch.diag(x.eps[:o]) + E("ne,mnie->mi", x.t1, x.ooov) + 0.5 * E("inef,mnef->mi", h.tau, x.oovv)
    h.Fae = torch.diag(x.eps[o:]) - E("mf,maef->ae", x.t1, x.ovvv) - 0.5 * E("mnaf,mnef->ae", h.tau, x.oovv)
    h.Y = E("jnfb,mnef->mbej", x.t2, x.oovv)
    h.Wmbej = (-x.ovov.transpose(2, 3) + E("jf,mbef->mbej", x.t1, x.ovvv) + E("nb,mnje->mbej", x.t1, x.ooov) - h.Y
               - E("nb,mnej->mbej", x.t1, E("jf,mnef->mnej", x.t1, x.oovv)))
    return h


def _anti(w):
    """w_ij - w_ji in the last two indices"""
    return w - w.transpose(-1, -2)


class _Ip:
    def __init__(self, x):
        h = _common(x)
        self.x, self.h, self.o, self.v = x, h, x.o, x.v
        h.Wmnij = x.oooo + _anti(E("je,mnie->mnij", x.t1, x.ooov)) + 0.5 * E("ijef,mnef->mnij", h.tau, x.oovv)
        h.Wmnie = x.ooov + E("if,mnfe->mnie", x.t1, x.oovv)
        X = -x.ovov.transpose(2, 3) - h.Y
        h.Wmbij = (x.ooov.permute(2, 3, 0, 1) - E("me,ijbe->mbij", h.Fme, x.t2) - E("nb,mnij->mbij", x.t1, h.Wmnij)
                   + 0.5 * E("mbef,ijef->mbij", x.ovvv, h.tau) - _anti(E("mnje,inbe->mbij", x.ooov, x.t2))
                   + _anti(E("ie,mbej->mbij", x.t1, X)))
        a, b = _pairs(self.o)
        self.i, self.j = a, b

    def unpack(self, r):
        o, v = self.o, self.v
        full = r.new_zeros((len(r), o, o, v))
        p = r[:, o:].reshape(len(r), -1, v)
        full[:, self.i, self.j] = p
        full[:, self.j, self.i] = -p
        return r[:, :o], full

    def pack(self, s1, s2):
        return torch.cat([s1, s2[:, self.i, self.j].reshape(len(s1), -1)], 1)

    def sigma(self, r):
        x, h = self.x, self.h
        r1, r2 = self.unpack(r)
        s1 = -E("mi,zm->zi", h.Fmi, r1) + E("me,zime->zi", h.Fme, r2) - 0.5 * E("mnie,zmne->zi", h.Wmnie, r2)
        xe = E("mnef,zmnf->ze", x.oovv, r2)
        u = E("maei,zmje->zija", h.Wmbej, r2) - E("mi,zmja->zija", h.Fmi, r2)
        s2 = (-E("maij,zm->zija", h.Wmbij, r1) + E("ae,zije->zija", h.Fae, r2) + u - u.transpose(1, 2)
              + 0.5 * E("mnij,zmna->zija", h.Wmnij, r2) + 0.5 * E("ijae,ze->zija", x.t2, xe))
        return self.pack(s1, s2)

    def free(self, orb):
        """b_p"""
        o, x, rows = self.o, self.x, []
        for p in orb:
            if p < o:
                rows.append((torch.eye(o, dtype=torch.float64, device="cuda")[p], torch.zeros_like(x.t2[:, :, 0])))
            else:
                rows.append((x.t1[:, p - o], x.t2[:, :, p - o]))
        return self.pack(torch.stack([r[0] for r in rows]), torch.stack([r[1] for r in rows]))

    def left(self, orb):
        """c_q"""
        o, x, rows = self.o, self.x, []
        c1 = torch.eye(o, dtype=torch.float64, device="cuda") - x.t1 @ x.l1.T - 0.5 * E("inef,knef->ik", x.t2, x.l2)
        for q in orb:
            if q >= o:
                rows.append((x.l1[:, q - o], x.l2[:, :, q - o]))
                continue
            s = -E("e,klec->klc", x.t1[q], x.l2)
            s[q] += x.l1
            s[:, q] -= x.l1
            rows.append((c1[q], s))
        return self.pack(torch.stack([r[0] for r in rows]), torch.stack([r[1] for r in rows]))


class _Ea:
    def __init__(self, x):
        h = _common(x)
        self.x, self.h, self.o, self.v = x, h, x.o, x.v
        a, b = _pairs(self.v)
        self.i, self.j = a, b
        half = x.eps.new_zeros((self.v, self.v, len(a)))
        half[a, b] = x.vvvv
        half[b, a] = -x.vvvv
        vvvv = x.eps.new_zeros((self.v,) * 4)
        vvvv[:, :, a, b] = half
        vvvv[:, :, b, a] = -half
        pab = lambda w: w - w.transpose(0, 1)  # noqa: E731
        h.Wabef = (vvvv + pab(E("mb,maef->abef", x.t1, x.ovvv)) + 0.5 * E("mnab,mnef->abef", h.tau, x.oovv))
        h.Wamef = -x.ovvv.transpose(0, 1) - E("na,nmef->amef", x.t1, x.oovv)
        X = -x.ovov.transpose(2, 3) - E("njbf,mnef->mbej", x.t2, x.oovv)
        h.Wabej = (-x.ovvv.permute(2, 3, 1, 0) - E("me,mjab->abej", h.Fme, x.t2) + E("jf,abef->abej", x.t1, h.Wabef)
                   - 0.5 * E("mnje,mnab->abej", x.ooov, h.tau) - pab(E("mbef,mjaf->abej", x.ovvv, x.t2))
                   - pab(E("ma,mbej->abej", x.t1, X)))

    def unpack(self, r):
        o, v = self.o, self.v
        full = r.new_zeros((len(r), v, v, o))
        p = r[:, v:].reshape(len(r), -1, o)
        full[:, self.i, self.j] = p
        full[:, self.j, self.i] = -p
        return r[:, :v], full

    pack = _Ip.pack

    def sigma(self, r):
        x, h = self.x, self.h
        r1, r2 = self.unpack(r)
        s1 = E("ae,ze->za", h.Fae, r1) + E("me,zaem->za", h.Fme, r2) + 0.5 * E("amef,zefm->za", h.Wamef, r2)
        u = E("ae,zebj->zabj", h.Fae, r2) + E("mbej,zaem->zabj", h.Wmbej, r2)
        xm = E("mnef,zefn->zm", x.oovv, r2)
        s2 = (E("abej,ze->zabj", h.Wabej, r1) - E("mj,zabm->zabj", h.Fmi, r2) + u - u.transpose(1, 2)
              + 0.5 * E("abef,zefj->zabj", h.Wabef, r2) - 0.5 * E("mjab,zm->zabj", x.t2, xm))
        return self.pack(s1, s2)

    def free(self, orb):
        """b_q of virtual q: the unit 1p vectors"""
        s1 = torch.eye(self.v, dtype=torch.float64, device="cuda")[[q - self.o for q in orb]]
        return self.pack(s1, s1.new_zeros((len(orb), self.v, self.v, self.o)))

    def left(self, orb):
        """c_p of virtual p"""
        x, rows = self.x, []
        c1 = torch.eye(self.v, dtype=torch.float64, device="cuda") - E("ka,kc->ac", x.t1, x.l1)
        c1 = c1 - 0.5 * E("klad,klcd->ac", x.t2, x.l2)
        for p in orb:
            a = p - self.o
            s = -E("k,knef->efn", x.t1[:, a], x.l2)
            s[a] += x.l1.T
            s[:, a] -= x.l1.T
            rows.append((c1[a], s))
        return self.pack(torch.stack([r[0] for r in rows]), torch.stack([r[1] for r in rows]))


def _system(case, seed):
    """(operator, dense M, b rows, c rows, sign): the EA half is (w + i eta - M) y = b."""
    x = _inputs(case, seed)
    op = _Ea(x) if case.get("sector") == "ea" else _Ip(x)
    eye = torch.eye(_dim(case), dtype=torch.float64, device="cuda")
    M = torch.cat([op.sigma(e) for e in eye.split(512)]).T.contiguous()
    orb = _orbitals(case)
    return M, op.free(orb), op.left(orb), -1.0 if case.get("sector") == "ea" else 1.0


def _spectral(G):
    return -torch.diagonal(G, dim1=1, dim2=2).imag.sum(1) / math.pi


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sigma", "init"):
        op, X = _Ip(_inputs(case, seed)), _block(case, seed)
        if not case.get("transpose"):
            return torch.cat([torch.complex(op.sigma(r.real), op.sigma(r.imag)) for r in X.split(6)])
        if _dim(case) > LU_MAX:
            return None
        M = torch.cat([op.sigma(e) for e in torch.eye(_dim(case), dtype=torch.float64, device="cuda").split(512)]).T
        return torch.complex(X.real @ M, X.imag @ M)
    if _dim(case) > LU_MAX or kind == "spectrum":
        return None
    M, b, c, sign = _system(case, seed)
    bc, cc = b.T.to(torch.complex128), c.to(torch.complex128)
    eye = torch.eye(len(M), dtype=torch.complex128, device="cuda")

    def solve(w):
        return torch.linalg.solve(sign * M + (w - 1j * sign * case["eta"]) * eye, bc)

    if kind == "eval":   # Galerkin projection on the span of the solutions at the seeds
        V = torch.linalg.qr(torch.cat([solve(w) for w in _seeds(case)], 1))[0]
        Mh, bh, ch = V.mH @ (M.to(torch.complex128) @ V), V.mH @ bc, cc @ V
        one = torch.eye(len(Mh), dtype=torch.complex128, device="cuda")
        G = torch.stack([(ch @ torch.linalg.solve(Mh + (w - 1j * case["eta"]) * one, bh)).T for w in _freqs(case, seed)])
        return {"G": G, "A": _spectral(G)}
    xs = [solve(w) for w in _freqs(case, seed)]
    G = torch.stack([(cc @ x).T for x in xs])
    if kind == "gradient":
        return {"G": G, "g": None}
    return {"G": G, "X": torch.stack([x.T for x in xs]) if case["vectors"] else None}

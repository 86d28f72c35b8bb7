"""What users of this library have it compute, as cases that can be timed.

Each case is one call, or one short chain of calls, of the public entry points
(paper_2212_06635_gb300.tm, the binding of include/tm.h) on a lattice held in a
tm_ctx, as a hybrid Monte Carlo program would issue it:

  apply       one operator application on a native field (what every solver does
              hundreds of times per solve), in all storage precisions
  apply_dw    the operator of the reliable updates (double-word arithmetic on FP64 fields)
  force       the hopping term's outer products of all pairs of a rational monomial
  refresh     a new gauge field: load it, rebuild the clover term and its inverses,
              and apply the first operator (which makes the low-precision copies)
  solve_cg    one mixed-precision CG solve of the light doublet
  multishift  one multishift solve of the heavy doublet with shift-by-shift refinement
  ptc         one application of the learned preconditioner

Lattices, couplings, the shift range and the network's channels are those of the
repository's own workloads; extents between them are generic.  Inputs are seeded
synthetic fields: SU(3) links U = exp(i eps H) with a plaquette near 0.59 and
complex Gaussian spinors, made on the GPU.

`exact` recomputes a case in plain torch FP64 / complex128 from the definitions
in include/tm.h, independent of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2212_06635_gb300 import tm

DEV = "cuda"
CSW = 1.69
EPS = 0.2197              # width of the link distribution: mean plaquette 0.590
PREC = {"f64": tm.TM_F64, "f32": tm.TM_F32, "bf16": tm.TM_BF16, "f16": tm.TM_F16}
OPS = {"MDAGM": tm.TM_MDAGM, "QPQM": tm.TM_QPQM, "QH_SQ": tm.TM_QH_SQ, "QHAT_PLUS": tm.TM_QHAT_PLUS,
       "QHAT_MINUS": tm.TM_QHAT_MINUS, "QH": tm.TM_QH, "QH_DAG": tm.TM_QH_DAG}
HEAVY = ("QH", "QH_DAG", "QH_SQ")
# factors of each operator as signs, the first applied first (include/tm.h)
SIGNS = {"MDAGM": (+1, -1), "QPQM": (-1, +1), "QH_SQ": (-1, +1), "QHAT_PLUS": (+1,), "QHAT_MINUS": (-1,),
         "QH": (+1,), "QH_DAG": (-1,)}
LIGHT = dict(kappa=0.1400, mu=0.0015, mubar=0.0, epsbar=0.0)
DOUBLET = dict(kappa=0.1400, mu=0.0, mubar=0.1246, epsbar=0.1350)
BOTH = dict(kappa=0.1400, mu=0.0015, mubar=0.1246, epsbar=0.1350)
NETWORK = dict(kappa=0.1394265, mu=0.00072, mubar=0.0, epsbar=0.0)
CHANNELS = (1, 8, 8, 8, 1)
LAMBDA_MAX = 2.75         # 1.02 x the power-iteration bound of Q_h Q_h^dagger on such fields
# A solve's x is FP64 and is stated by its residual; 1e-12 is the tolerance of the
# repository's 4^4 workload and leaves x itself determined to about 1e-11.
TOL = 1e-12


def _case(name, kind, dims, **kw):
    d = dict(name=name, kind=kind, X=dims[0], Y=dims[1], Z=dims[2], T=dims[3])
    d.update(kw)
    return d


def listed():
    return [
        # the smallest members of the uneven batch: launches and latency count
        _case("apply_light_f32_8x16", "apply", (8, 8, 8, 16), op="MDAGM", prec="f32"),
        # the inner operator of the mixed-precision CG on the benchmark lattice
        _case("apply_light_f16_32x64", "apply", (32, 32, 32, 64), op="MDAGM", prec="f16"),
        # an uneven lattice, the other ordering of the factors (the HMC's), BF16 storage
        _case("apply_light_bf16_uneven", "apply", (18, 22, 26, 44), op="QPQM", prec="bf16"),
        # the inner operators of the heavy doublet's multishift solve and of its refinement
        _case("apply_heavy_f32_24x48", "apply", (24, 24, 24, 48), op="QH_SQ", prec="f32"),
        _case("apply_heavy_f16_24x48", "apply", (24, 24, 24, 48), op="QH_SQ", prec="f16"),
        # plain FP64: the final residual of every solve, the power iteration, FP64 CG
        _case("apply_light_f64_16x32", "apply", (16, 16, 16, 32), op="MDAGM", prec="f64"),
        # the true residual at a reliable update
        _case("apply_dw_light_24x48", "apply_dw", (24, 24, 24, 48), op="MDAGM"),
        # the force of a rational monomial: 12 two-flavour pairs on every link
        _case("force_heavy_f32_24x48", "force", (24, 24, 24, 48), prec="f32", flavours=2, pairs=12, gamma5=True),
        # every step of a trajectory: a new gauge field up to the first operator result
        _case("refresh_24x48", "refresh", (24, 24, 24, 48), op="QH_SQ", prec="f32"),
        # whole solves: light mixed-precision CG; the heavy doublet's 12 shifts
        _case("solve_cg_f16_32x64", "solve_cg", (32, 32, 32, 64), op="MDAGM", sloppy="f16"),
        _case("multishift_f32_24x48", "multishift", (24, 24, 24, 48), shifts=12, sloppy="f32", refine="f32"),
        # the learned preconditioner's application inside flexible CG
        _case("ptc_apply_24x48", "ptc", (24, 24, 24, 48)),
    ]


def _dims(rng, lo, hi):
    """Even extents with a volume spread over the logarithm of lo .. hi sites, T the longest."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        s = (v / 2.0) ** 0.25
        d = [max(4, 2 * int(round(s * math.exp(rng.uniform(-0.3, 0.3)) / 2))) for _ in range(3)]
        t = 2 * int(round(v / (d[0] * d[1] * d[2]) / 2))
        if t >= 4 and lo <= d[0] * d[1] * d[2] * t <= hi:
            return (*d, t)


def draw(rng):
    case = _drawn(rng)
    del case["name"]
    return case


def _drawn(rng):
    kind = rng.choice(["apply"] * 5 + ["apply_dw", "force", "refresh", "solve_cg", "multishift", "ptc"])
    v24, v32 = 24 ** 3 * 48, 32 ** 3 * 64
    if kind == "apply":
        heavy = rng.random() < 0.4
        prec = rng.choice(["f16", "f16", "f32", "f32", "bf16", "f64"])
        op = rng.choice(list(HEAVY) if heavy else ["MDAGM", "QPQM", "QHAT_PLUS", "QHAT_MINUS"])
        hi = 16 ** 3 * 32 if prec == "f64" else (v24 if heavy else v32)
        return _case("", kind, _dims(rng, 512, hi), op=op, prec=prec)
    if kind == "apply_dw":
        op = rng.choice(["MDAGM", "QPQM", "QH_SQ"])
        return _case("", kind, _dims(rng, 4096, v24 if op != "QH_SQ" else v24 // 2), op=op)
    if kind == "force":
        return _case("", kind, _dims(rng, 4096, v24), prec=rng.choice(["f32", "f16", "bf16"]),
                     flavours=rng.choice([1, 2]), pairs=rng.randint(1, 12), gamma5=rng.random() < 0.7)
    if kind == "refresh":
        return _case("", kind, _dims(rng, 4096, v24), op=rng.choice(["MDAGM", "QH_SQ"]),
                     prec=rng.choice(["f32", "f16"]))
    if kind == "solve_cg":
        return _case("", kind, _dims(rng, 4096, v24), op=rng.choice(["MDAGM", "QPQM"]),
                     sloppy=rng.choice(["f16", "f16", "f16", "f32", "f32", "f64"]))
    if kind == "multishift":
        return _case("", kind, _dims(rng, 4096, v24 // 2), shifts=rng.randint(3, 12), sloppy="f32",
                     refine=rng.choice(["f32", "f16"]))
    return _case("", kind, _dims(rng, 4096, v24))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, part):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + part) % (1 << 62))
    return g


def _dims_of(case):
    return case["X"], case["Y"], case["Z"], case["T"]


def _links(case, seed):
    """Canonical links [site][mu][3][3] (complex128): U = exp(i eps H), then reunitarised in FP64."""
    n = 4 * math.prod(_dims_of(case))
    h = torch.randn((n, 8), generator=_gen(seed, 1), device=DEV)
    m = torch.zeros((n, 3, 3), dtype=torch.complex64, device=DEV)
    r3 = 1.0 / math.sqrt(3.0)
    for (a, b), (p, q) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        m[:, a, b] = torch.complex(h[:, p], -h[:, q])
        m[:, b, a] = torch.complex(h[:, p], h[:, q])
    m[:, 0, 0] = h[:, 2] + r3 * h[:, 7]
    m[:, 1, 1] = -h[:, 2] + r3 * h[:, 7]
    m[:, 2, 2] = -2.0 * r3 * h[:, 7]
    m *= 1j * EPS / 4.0
    one = torch.eye(3, dtype=torch.complex64, device=DEV)
    u = one + m / 6.0
    for k in (5, 4, 3, 2, 1):
        u = one + _mul3(m, u) / k
    u = _mul3(u, u)
    u = _mul3(u, u).to(torch.complex128)
    r0 = u[:, 0] / u[:, 0].abs().square().sum(-1, keepdim=True).sqrt()
    r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=1).reshape(n // 4, 4, 3, 3).contiguous()


def _mul3(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _spinor(case, seed, part, flavours):
    """Canonical half-lattice field [site][(flavour)][spin][colour], Gaussian re and im."""
    n = math.prod(_dims_of(case)) // 2
    f = torch.randn((n, flavours, 4, 3, 2), generator=_gen(seed, part), device=DEV, dtype=torch.float64)
    return torch.view_as_complex(f)


def _action(case):
    if case["kind"] == "refresh":
        return BOTH
    if case["kind"] == "ptc":
        return NETWORK
    heavy = case["kind"] == "multishift" or case.get("op") in HEAVY or case.get("flavours") == 2
    return DOUBLET if heavy else LIGHT


def _flavours(case):
    return case.get("flavours") or (2 if case["kind"] == "multishift" or case.get("op") in HEAVY else 1)


def _shifts(case):
    n = case["shifts"]
    return [LAMBDA_MAX * 10.0 ** (-5.0 + 5.0 * k / (n - 1)) for k in range(n)]


def _weights(seed):
    """A network near the identity, with noise, as its training starts from (canonical layout)."""
    rng = np.random.default_rng(seed)
    out = []
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        w = 0.03 * (rng.uniform(-1, 1, (9, co, ci, 4, 4)) + 1j * rng.uniform(-1, 1, (9, co, ci, 4, 4)))
        for a in range(min(ci, co)):
            w[0, a, a] += 0.5 * np.eye(4)
        out.append(w.astype(np.complex64).astype(np.complex128))
    return out


class State:
    """A context with its gauge field and clover term, and a case's fields; gives the memory back when dropped."""

    def __init__(self, case):
        self.case = case
        self.net = None
        self.ctx = tm.tm_create(_dims_of(case))

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.net is not None:
                tm.tm_ptc_destroy(self.net)
            tm.tm_destroy(self.ctx)
        except Exception:
            pass


def _native(s, prec, flavours, canonical=None):
    f = torch.empty(tm.tm_field_bytes(s.ctx, prec, flavours), dtype=torch.uint8, device=DEV)
    if canonical is not None:
        tm.tm_field_import(s.ctx, prec, flavours, f, canonical)
    return f


def prepare(case, seed):
    kind, act = case["kind"], _action(case)
    s = State(case)
    s.links = _links(case, seed)
    tm.tm_gauge_load(s.ctx, s.links, float(seed))
    tm.tm_clover_compute(s.ctx, csw=CSW, bc_t=-1, **act)
    nf = _flavours(case)
    if kind in ("apply", "apply_dw", "refresh"):
        p = PREC[case.get("prec", "f64")]
        s.x = _native(s, p, nf, _spinor(case, seed, 2, nf))
        s.out = _native(s, p, nf)
    elif kind == "force":
        p = PREC[case["prec"]]
        s.coeff = [0.1 / (k + 1) for k in range(case["pairs"])]
        fields = [_native(s, p, nf, _spinor(case, seed, 10 + j, nf)) for j in range(4 * case["pairs"])]
        s.xs = [(fields[4 * k], fields[4 * k + 1]) for k in range(case["pairs"])]
        s.ys = [(fields[4 * k + 2], fields[4 * k + 3]) for k in range(case["pairs"])]
        s.force = torch.zeros((math.prod(_dims_of(case)), 4, 3, 3), dtype=torch.complex128, device=DEV)
    elif kind in ("solve_cg", "multishift"):
        s.b = _spinor(case, seed, 2, nf).contiguous()
        s.sp = tm.solve_params(tol=TOL, sloppy=PREC[case["sloppy"]], refine=PREC[case.get("refine", "f64")])
        n = case.get("shifts", 1)
        s.x = [torch.zeros_like(s.b) for _ in range(n)]
    else:
        s.net = tm.tm_ptc_create(CHANNELS)
        tm.tm_ptc_set_weights(s.net, np.concatenate([w.ravel() for w in _weights(seed)]))
        s.x = _native(s, tm.TM_F32, 1, _spinor(case, seed, 2, 1))
        s.out = _native(s, tm.TM_F32, 1)
    if kind != "refresh":
        s.links = None          # the context keeps its own copy
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _values(case, out, prec, nf):
    """A native field as its values.  A 16-bit field's per-site FP32 scale is returned in the
    field's own 16 bits: its values carry no more than that."""
    n = 24 * nf * (math.prod(_dims_of(case)) // 2)
    if prec == "f64":
        return out.view(torch.float64)
    if prec == "f32":
        return out.view(torch.float32)
    t = torch.float16 if prec == "f16" else torch.bfloat16
    return {"stored": out[:2 * n].view(t), "scale": out[2 * n:].view(torch.float32).to(t)}


def run(s):
    case = s.case
    kind, nf = case["kind"], _flavours(case)
    if kind == "apply":
        tm.tm_apply_Mhat(s.ctx, OPS[case["op"]], PREC[case["prec"]], s.out, s.x)
        return _values(case, s.out, case["prec"], nf)
    if kind == "apply_dw":
        tm.tm_apply_Mhat_dw(s.ctx, OPS[case["op"]], s.out, s.x)
        return _values(case, s.out, "f64", nf)
    if kind == "force":
        tm.tm_force_outer(s.ctx, PREC[case["prec"]], nf, s.coeff, s.xs, s.ys, s.force, gamma5_y=case["gamma5"])
        return s.force
    if kind == "refresh":
        tm.tm_gauge_load(s.ctx, s.links, tm.tm_gauge_id(s.ctx) + 1.0)
        tm.tm_clover_compute(s.ctx, csw=CSW, bc_t=-1, **_action(case))
        tm.tm_apply_Mhat(s.ctx, OPS[case["op"]], PREC[case["prec"]], s.out, s.x)
        return _values(case, s.out, case["prec"], nf)
    if kind == "solve_cg":
        s.x[0].zero_()
        tm.tm_solve_cg(s.ctx, OPS[case["op"]], s.sp, s.x[0], s.b)
        return s.x[0]
    if kind == "multishift":
        tm.tm_solve_multishift(s.ctx, tm.TM_QH_SQ, _shifts(case), s.x, s.b, s.sp)
        return list(s.x)
    tm.tm_ptc_apply(s.net, s.ctx, s.out, s.x)
    return _values(case, s.out, "f32", 1)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Inputs once, outputs once, in the storage the call names; links count 12 reals where 12 are kept."""
    kind, nf = case["kind"], _flavours(case)
    v = math.prod(_dims_of(case))
    vh = v // 2
    esz = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}

    def operator(prec, factors):
        e = esz[prec]
        link = 18 if prec in ("f64", "bf16") else 12
        spin = 24 * nf * e + (4 if e == 2 else 0)
        nb = vh * (2 * spin + 8 * link * e + (144 + 72) * e)          # in, out, links, inverse, clover
        return nb, factors * vh * nf * 3792.0

    if kind == "apply":
        b, f = operator(case["prec"], len(SIGNS[case["op"]]))
    elif kind == "apply_dw":
        b, f = operator("f64", 2)
    elif kind == "force":
        e, n = esz[case["prec"]], case["pairs"]
        b = 2 * n * v * (24 * nf * e + (4 if e == 2 else 0)) + 4 * v * 12 * 4 + 2 * 4 * v * 18 * 8
        f = 4.0 * v * (n * nf * (4 * 24 + 36 * 8) + 300)
    elif kind == "refresh":
        nb, f = operator(case["prec"], 2)
        b = v * 4 * 18 * 8 + nb + vh * (2 * 72 + 288) * 8             # links, FP64 clover terms and inverses
        f += v * 6 * (12 * 198.0) + vh * 2 * 4 * 1500.0
    elif kind in ("solve_cg", "multishift"):
        # about 220 iterations on such fields, each streaming the operator's links and
        # clover once and its vectors; the shifts' directions and solutions once a solve
        nb, f = operator(case["sloppy"], 2)
        its, n = 220, case.get("shifts", 1)
        b = its * nb + (n + 1) * vh * 24 * nf * 8
        f = its * (f + vh * nf * 24 * 2.0 * (3 + 2 * (n if kind == "multishift" else 1)))
    else:
        pairs = list(zip(CHANNELS[:-1], CHANNELS[1:]))
        b = 2 * vh * 24 * 4 + v * 4 * 12 * 2                          # FP32 field in and out, links
        f = float(sum(v * (8 * ci * 4 * 66.0 + 9 * ci * co * 3 * 16 * 8.0) for ci, co in pairs))
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
class Lattice:
    """Definitions of include/tm.h on half-lattice fields [flavour][spin][colour][site]."""

    def __init__(self, case, seed, clover=True):
        self.dims = X, Y, Z, T = _dims_of(case)
        self.V = X * Y * Z * T
        act = _action(case)
        self.kappa = act["kappa"]
        self.mu, self.mubar, self.eps = (2 * self.kappa * act[k] for k in ("mu", "mubar", "epsbar"))
        lex = torch.arange(self.V, device=DEV)
        c = [lex % X, (lex // X) % Y, (lex // (X * Y)) % Z, lex // (X * Y * Z)]
        st = (1, X, X * Y, X * Y * Z)
        par = (c[0] + c[1] + c[2] + c[3]) % 2
        self.sites = [torch.nonzero(par == p).ravel() for p in (0, 1)]
        self.fwd = [torch.where(c[m] + 1 == self.dims[m], lex - (self.dims[m] - 1) * st[m], lex + st[m]) for m in range(4)]
        self.bwd = [torch.where(c[m] == 0, lex + (self.dims[m] - 1) * st[m], lex - st[m]) for m in range(4)]
        one = torch.ones(self.V, dtype=torch.float64, device=DEV)
        self.ph_f = torch.where(c[3] + 1 == T, -one, one)
        self.ph_b = torch.where(c[3] == 0, -one, one)
        self.U = _links(case, seed).permute(1, 2, 3, 0).contiguous()      # [mu][3][3][site]
        if clover:
            self._clover()

    @staticmethod
    def mm(a, b):
        out = torch.empty_like(a)
        for i in range(3):
            for j in range(3):
                out[i, j] = a[i, 0] * b[0, j]
                for k in (1, 2):
                    out[i, j].addcmul_(a[i, k], b[k, j])
        return out

    @staticmethod
    def dg(a):
        return a.transpose(0, 1).conj().resolve_conj()

    def _clover(self):
        mm, dg = self.mm, self.dg
        F = {}
        for m in range(4):
            for n in range(m + 1, 4):
                um, un = self.U[m], self.U[n]
                xm, xn, ym, yn = self.fwd[m], self.fwd[n], self.bwd[m], self.bwd[n]
                q = mm(mm(um, un[..., xm]), dg(mm(un, um[..., xn])))
                q += mm(mm(un, dg(um[..., xn[ym]])), mm(dg(un[..., ym]), um[..., ym]))
                q += mm(dg(mm(un[..., yn[ym]], um[..., ym])), mm(um[..., yn[ym]], un[..., yn]))
                q += mm(mm(dg(un[..., yn]), um[..., yn]), mm(un[..., xm[yn]], dg(um)))
                f = (q - dg(q)) / 8.0
                tr = (f[0, 0] + f[1, 1] + f[2, 2]) / 3.0
                for k in range(3):
                    f[k, k] -= tr
                F[m, n] = f
        k = self.kappa * CSW
        self.A = []                                                       # per parity [chirality][6][6][site]
        for p in (0, 1):
            s = self.sites[p]
            a = torch.zeros((2, 6, 6, s.numel()), dtype=torch.complex128, device=DEV)
            for c, sg in ((0, 1.0), (1, -1.0)):
                a1 = (F[1, 2] + sg * F[0, 3])[..., s]
                a2 = (sg * F[1, 3] - F[0, 2])[..., s]
                a3 = (F[0, 1] + sg * F[2, 3])[..., s]
                a[c, :3, :3] = -1j * k * a3
                a[c, 3:, 3:] = 1j * k * a3
                a[c, :3, 3:] = -k * (1j * a1 + a2)
                a[c, 3:, :3] = -k * (1j * a1 - a2)
                for r in range(6):
                    a[c, r, r] += 1.0
            self.A.append(a)

    def local(self, p, heavy, sign):
        """The site-local matrix of parity p per chirality: 6 x 6, or 12 x 12 over both flavours."""
        a = self.A[p]
        n = 12 if heavy else 6
        out = torch.zeros((2, n, n, a.shape[-1]), dtype=torch.complex128, device=DEV)
        for c, sg in ((0, 1.0), (1, -1.0)):
            for f in range(n // 6):
                out[c, 6 * f:6 * f + 6, 6 * f:6 * f + 6] = a[c]
                for r in range(6):
                    tw = self.mubar * (1 - 2 * f) if heavy else self.mu
                    out[c, 6 * f + r, 6 * f + r] += 1j * sign * sg * tw
                    if heavy:
                        out[c, 6 * f + r, 6 * (1 - f) + r] -= self.eps
        return out

    @staticmethod
    def block(m, psi):
        """Chirality blocks m on psi [flavour][4][3][site]."""
        nf, n = psi.shape[0], psi.shape[-1]
        v = psi.reshape(nf, 2, 6, n).transpose(0, 1).reshape(2, 6 * nf, n)
        w = torch.empty_like(v)
        for r in range(6 * nf):
            w[:, r] = (m[:, r] * v).sum(1)
        return w.reshape(2, nf, 6, n).transpose(0, 1).reshape(nf, 4, 3, n)

    def _tables(self, p):
        """Neighbour indices and links of the hops that end on parity p."""
        if not hasattr(self, "tab"):
            self.tab = {}
        if p not in self.tab:
            s = self.sites[p]
            t = []
            for m in range(4):
                f, b = self.fwd[m][s], self.bwd[m][s]
                uf, ub = self.U[m][..., s].clone(), self.dg(self.U[m][..., b]).clone()
                if m == 3:
                    uf *= self.ph_f[s]
                    ub *= self.ph_b[s]
                t.append((f // 2, uf, b // 2, ub))
            self.tab[p] = t
        return self.tab[p]

    def hop(self, p, psi):
        """H psi on the sites of parity p, psi on the other parity."""
        out = torch.zeros_like(psi)
        up, dn = out[:, :2], out[:, 2:]
        for m, (fi, uf, bi, ub) in enumerate(self._tables(p)):
            for s, idx, u in ((-1.0, fi, uf), (+1.0, bi, ub)):
                q = psi[..., idx]
                a, b, c, d = q[:, 0], q[:, 1], q[:, 2], q[:, 3]
                if m == 0:
                    h = (a - 1j * s * d, b - 1j * s * c)
                elif m == 1:
                    h = (a - s * d, b + s * c)
                elif m == 2:
                    h = (a - 1j * s * c, b + 1j * s * d)
                else:
                    h = (a - s * c, b - s * d)
                h = torch.stack(h, 1)                                     # [flavour][2][3][site]
                g = u[:, 0] * h[:, :, 0, None]
                for k in (1, 2):
                    g = torch.addcmul(g, u[:, k].expand_as(g), h[:, :, k, None].expand_as(g))
                up += g
                if m == 0:
                    dn += s * 1j * g.flip(1)
                elif m == 1:
                    dn[:, 0] += s * g[:, 1]
                    dn[:, 1] -= s * g[:, 0]
                elif m == 2:
                    dn[:, 0] += s * 1j * g[:, 0]
                    dn[:, 1] -= s * 1j * g[:, 1]
                else:
                    dn -= s * g
        return out

    def operators(self, heavy, signs):
        """The Schur operators of these signs as functions."""
        odd = {s: self.local(1, heavy, s) for s in set(signs)}
        inv = {}
        for s in set(signs):
            m = self.local(0, heavy, s).permute(3, 0, 1, 2).contiguous()
            inv[s] = torch.linalg.inv(m).permute(1, 2, 3, 0).contiguous()

        def q(s, psi):
            t = self.block(inv[s], self.hop(0, psi))
            w = self.block(odd[s], psi) - self.kappa ** 2 * self.hop(1, t)
            w[:, 2:] *= -1.0
            return w

        return q


def _soa(canonical):
    return canonical.permute(1, 2, 3, 0).contiguous()                     # [flavour][spin][colour][site]


def _exact_native(psi, prec):
    """The reals of psi in the native order of a storage precision."""
    n = psi.shape[-1]
    r = torch.view_as_real(psi.reshape(-1, n).contiguous()).permute(0, 2, 1).reshape(-1, n)   # [real][site]
    if prec in ("f16", "bf16"):
        scale = r.abs().amax(0)
        r = r / scale
    w = {"f64": 2, "f32": 4, "f16": 8, "bf16": 8}[prec]
    flat = r.reshape(-1, w, n).permute(0, 2, 1).reshape(-1)
    return {"stored": flat, "scale": scale} if prec in ("f16", "bf16") else flat


def _exact_force(case, seed):
    lat = Lattice(case, seed, clover=False)
    nf, V = case["flavours"], lat.V
    full = torch.empty((4, nf, 4, 3, V), dtype=torch.complex128, device=DEV)
    W = torch.zeros((4, 3, 3, V), dtype=torch.complex128, device=DEV)
    # (1 + s gamma) B = (h, s G^+ h): sums over spin of A (x) ((1 + s gamma) B)^* run over two components
    def half(f, m, s):
        a, b, c, d = f[:, 0], f[:, 1], f[:, 2], f[:, 3]
        if m == 0:
            return a - 1j * s * d, b - 1j * s * c
        if m == 1:
            return a - s * d, b + s * c
        if m == 2:
            return a - 1j * s * c, b + 1j * s * d
        return a - s * c, b - s * d

    for k in range(case["pairs"]):
        for j in range(2):
            for p in (0, 1):
                full[j][..., lat.sites[p]] = _soa(_spinor(case, seed, 10 + 4 * k + 2 * j + p, nf))
        X, Yk = full[0], full[1]
        if case["gamma5"]:
            Yk = Yk.clone()
            Yk[:, 2:] *= -1.0
        for m in range(4):
            xn, yn = X[..., lat.fwd[m]], Yk[..., lat.fwd[m]]
            for u, v in ((half(xn, m, -1.0), half(Yk, m, -1.0)), (half(yn, m, 1.0), half(X, m, 1.0))):
                for l in range(2):
                    for f in range(nf):
                        W[m] += (0.1 / (k + 1)) * (u[l][f][:, None] * v[l][f][None].conj())
    W[3] *= lat.ph_f
    out = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device=DEV)
    for m in range(4):
        z = lat.mm(lat.U[m], W[m])
        z = 0.5 * (z - lat.dg(z))
        tr = (z[0, 0] + z[1, 1] + z[2, 2]) / 3.0
        for k in range(3):
            z[k, k] -= tr
        out[:, m] = z.permute(2, 0, 1)
    return out


def _exact_ptc(case, seed):
    lat = Lattice(case, seed, clover=False)
    phi = torch.zeros((1, 4, 3, lat.V), dtype=torch.complex128, device=DEV)
    phi[..., lat.sites[1]] = _soa(_spinor(case, seed, 2, 1).to(torch.complex64).to(torch.complex128))
    for w in _weights(seed):
        w = torch.from_numpy(w).to(DEV)
        co, ci = w.shape[1:3]
        out = torch.zeros((co * 4, 3 * lat.V), dtype=torch.complex128, device=DEV)
        for p in range(9):
            m = (p - 1) & 3
            if p == 0:
                t = phi
            else:
                f = phi[..., lat.fwd[m] if p <= 4 else lat.bwd[m]]
                u = lat.U[m] if p <= 4 else lat.dg(lat.U[m][..., lat.bwd[m]])
                if m == 3:
                    u = u * (lat.ph_f if p <= 4 else lat.ph_b)
                t = u[:, 0] * f[:, :, 0, None]
                for k in (1, 2):
                    t = torch.addcmul(t, u[:, k].expand_as(t), f[:, :, k, None].expand_as(t))
            out += w[p].permute(0, 2, 1, 3).reshape(co * 4, ci * 4) @ t.reshape(ci * 4, 3 * lat.V)
        phi = out.reshape(co, 4, 3, lat.V)
    return _exact_native(phi[..., lat.sites[1]], "f32")


def _dot(a, b):
    return torch.linalg.vecdot(a.reshape(-1), b.reshape(-1)).real


def _exact_solve(A, b, shifts, tol):
    """Textbook multishift CG in FP64: (A + s_k) x_k = b."""
    x = [torch.zeros_like(b) for _ in shifts]
    ps = [b.clone() for _ in shifts]
    r, p = b.clone(), b.clone()
    rr = bb = float(_dot(r, r))
    n = len(shifts)
    z, zo, al, be = [1.0] * n, [1.0] * n, 1.0, 0.0
    live = list(range(n))
    for _ in range(3000):
        ap = A(p) + shifts[0] * p
        alpha = rr / float(_dot(p, ap))
        for k in live:
            d = shifts[k] - shifts[0]
            zn = z[k] * zo[k] * al / (alpha * be * (zo[k] - z[k]) + zo[k] * al * (1 + d * alpha))
            x[k] += alpha * zn / z[k] * ps[k]
            zo[k], z[k] = z[k], zn
        r -= alpha * ap
        new = float(_dot(r, r))
        be_new = new / rr
        live = [k for k in live if z[k] * z[k] * new > tol * tol * bb]
        if not live:
            break
        p = r + be_new * p
        for k in live:
            ps[k] = z[k] * r + be_new * (z[k] / zo[k]) ** 2 * ps[k]
        rr, al, be = new, alpha, be_new
    return x


def exact(case, seed):
    kind, nf = case["kind"], _flavours(case)
    heavy = nf == 2
    if kind == "force":
        return _exact_force(case, seed)
    if kind == "ptc":
        return _exact_ptc(case, seed)
    lat = Lattice(case, seed)
    signs = SIGNS[case.get("op", "QH_SQ")]
    q = lat.operators(heavy, signs)
    b = _spinor(case, seed, 2, nf)
    if kind in ("apply", "apply_dw", "refresh"):
        psi = _soa(b)
        for s in signs:
            psi = q(s, psi)
        return _exact_native(psi, case.get("prec", "f64"))

    def A(psi):
        return q(signs[1], q(signs[0], psi))

    shifts = _shifts(case) if kind == "multishift" else [0.0]
    x = _exact_solve(A, _soa(b), shifts, 1e-14)
    x = [v.permute(3, 0, 1, 2).contiguous() for v in x]
    return x if kind == "multishift" else x[0]

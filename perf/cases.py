"""The work that users of this library have it do, as cases that can be timed.

Each case is one call (or the few calls that belong together) through the
public entry points of ``paper_1411_4439_gb300``: the multi-rhs Dslash and the
operators built from it, loading a gauge field, the bilinears, and the whole
solves. ``listed`` names the cases, ``draw`` gives more of the same ranges,
``prepare`` makes what a program has in hand before the call, ``run`` is one
pass and ``exact`` the same result from plain torch in 64 bits.

Lattices, bundle sizes, storage types and link compressions are those of the
library's configurations and tests. The solves run at m = 0.05 (0.01 for the
FP32 bundle): the lighter masses of the configurations take the same
iterations many times over and would need seconds a pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1411_4439_gb300 as H
from paper_1411_4439_gb300 import autograd as A

FAT, NAIK = 0.9, -1.0 / 24.0
PRECS = {"f64": H.HISQ_F64, "f32": H.HISQ_F32, "f16": H.HISQ_F16}
REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2}
ROWS = [1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 16]   # bundle sizes the per-rhs layouts take
CHUNK = {"f32": 2, "f16": 4}               # rhs in a 16-byte chunk of the bundle layout
OPS = {"M": H.HISQ_OP_M, "Mdag": H.HISQ_OP_MDAG, "dM": H.HISQ_OP_DM_DMU, "d2M": H.HISQ_OP_D2M_DMU2}
FLOPS = 1146                               # of one Dslash, per output site and rhs


def listed():
    return [
        # the smallest solve: FP64, one rhs, 8^4; a chain of tiny launches
        dict(name="cg f64 8^4 n1", kind="cg", prec="f64", L="8,8,8,8", n=1, ru=18, rn=18, mass=0.05,
             every=50, source="z2"),
        # the FP32 bundle solve with FP64 reliable updates
        dict(name="cg f32 32^3x8 n8", kind="cg", prec="f32", L="32,32,32,8", n=8, ru=18, rn=14, mass=0.01,
             every=50, source="z2"),
        # the mixed-precision bundle solve: 16-bit storage, FP64 reliable updates
        dict(name="cg f16 48^3x12 n8", kind="cg", prec="f16", L="48,48,48,12", n=8, ru=18, rn=14, mass=0.05,
             every=150, source="gauss"),
        # solves on several gauge fields of uneven volume in one call
        dict(name="batched f16 3 fields", kind="batched", prec="f16", L="24,24,24,6", n=16, L2="32,32,32,8", n2=8,
             L3="64,64,64,16", n3=4, ru=18, rn=14, mass=0.05, every=150, source="z2"),
        # forward and backward of the differentiable solve at mu != 0
        dict(name="grad f64 16^4 n4", kind="grad", prec="f64", L="16,16,16,16", n=4, ru=18, rn=18, mass=0.05, mu=0.1,
             source="z2"),
        # one hopping term on the solver's layout, 16-bit storage
        dict(name="dslash f16 bundle 48^3x12 n8", kind="dslash", prec="f16", layout="bundle", L="48,48,48,12", n=8,
             ru=18, rn=14, mu=0.0, parity=0, source="gauss"),
        # the same in FP32 on the largest lattice
        dict(name="dslash f32 bundle 64^3x16 n4", kind="dslash", prec="f32", layout="bundle", L="64,64,64,16", n=4,
             ru=18, rn=14, mu=0.0, parity=1, source="z2"),
        # the smallest call: one vector in the plain per-rhs layout
        dict(name="dslash f32 8^4 n1", kind="dslash", prec="f32", layout="aos", L="8,8,8,8", n=1, ru=18, rn=18,
             mu=0.0, parity=1, source="z2"),
        # the normal operator on a ragged lattice and an odd bundle, plain layout
        dict(name="mdagm f32 20x28x36x10 n6", kind="mdagm", prec="f32", L="20,28,36,10", n=6, ru=12, rn=14, mass=0.01,
             source="gauss"),
        # the full-lattice operator at mu != 0 in FP64, as the trace estimates use it
        dict(name="Mdag f64 24^3x6 n4", kind="apply", prec="f64", op="Mdag", L="24,24,24,6", n=4, ru=18, rn=18,
             mass=0.05, mu=0.1, source="z2"),
        # a new gauge field: load and compress its links, then the first Dslash on it
        dict(name="load f16 48^3x12", kind="load", prec="f16", L="48,48,48,12", n=8, ru=18, rn=14, source="gauss"),
        # the bilinears of the trace estimates
        dict(name="cdot f64 32^3x8 n16", kind="cdot", prec="f64", L="32,32,32,8", n=16, source="z2"),
    ]


def _draw_lattice(rng, vmin, vmax):
    """Even extents from 4 to 64, the volume spread over its logarithm."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    while True:
        ext = [2 * int(round(math.exp(rng.uniform(math.log(2), math.log(32))))) for _ in range(4)]
        v = math.prod(ext)
        if vmin <= v <= vmax and 0.7 * target <= v <= 1.4 * target:
            return ",".join(map(str, ext))


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "dslash", "cg", "cg", "mdagm", "apply", "load", "cdot", "grad", "batched"])
    prec = rng.choice(["f32", "f16"])
    ru, rn = rng.choice([(18, 18), (18, 14), (18, 14), (12, 14), (14, 14)])
    source = rng.choice(["z2", "gauss"])
    if kind == "dslash":
        layout = rng.choice(["bundle", "bundle", "aos", "soa"])
        if layout != "bundle" and rng.random() < 0.4:
            prec, ru, rn = "f64", 18, 18
        n = rng.choice([4, 8, 12, 16] if layout == "bundle" else ROWS)
        top = 8_000_000 * (4 if prec != "f64" else 1) // n
        return dict(kind=kind, prec=prec, layout=layout, L=_draw_lattice(rng, 4096, min(64 ** 3 * 16, top)), n=n, ru=ru,
                    rn=rn, mu=rng.choice([0.0, 0.0, 0.1]), parity=rng.randint(0, 1), source=source)
    if kind == "cg":
        mass = round(math.exp(rng.uniform(math.log(0.05), math.log(0.2))), 4)
        if rng.random() < 0.35:
            n = rng.randint(1, 4)
            return dict(kind=kind, prec="f64", L=_draw_lattice(rng, 4096, 65536), n=n, ru=18, rn=18, mass=mass, every=50,
                        source=source)
        n = rng.choice([1, 2, 3, 4, 6, 8, 8, 12, 16])
        return dict(kind=kind, prec=prec, L=_draw_lattice(rng, 4096, 8_000_000 // n), n=n, ru=ru, rn=rn, mass=mass,
                    every=rng.choice([50, 100, 150]), source=source)
    if kind == "batched":
        n, n2, n3 = (rng.choice([4, 8, 12, 16]) for _ in range(3))
        return dict(kind=kind, prec=prec, L=_draw_lattice(rng, 4096, 2_000_000 // n), n=n,
                    L2=_draw_lattice(rng, 4096, 2_000_000 // n2), n2=n2, L3=_draw_lattice(rng, 4096, 4_000_000 // n3),
                    n3=n3, ru=ru, rn=rn, mass=round(rng.uniform(0.05, 0.1), 3), every=150, source=source)
    if kind == "grad":
        return dict(kind=kind, prec="f64", L=_draw_lattice(rng, 4096, 65536), n=rng.randint(1, 4), ru=18, rn=18,
                    mass=round(rng.uniform(0.05, 0.15), 3), mu=round(rng.uniform(0.0, 0.15), 3), source=source)
    if kind == "mdagm":
        n = rng.choice([k for k in ROWS if k <= 12])
        return dict(kind=kind, prec=prec, L=_draw_lattice(rng, 4096, 8_000_000 // n), n=n, ru=ru, rn=rn,
                    mass=round(rng.uniform(0.002, 0.1), 4), source=source)
    if kind == "apply":
        if rng.random() < 0.6:
            prec, ru, rn = "f64", 18, 18
        n = rng.randint(1, 8)
        return dict(kind=kind, prec=prec, op=rng.choice(sorted(OPS)), L=_draw_lattice(rng, 4096, 2_000_000 // n), n=n,
                    ru=ru, rn=rn, mass=0.05, mu=round(rng.uniform(0.05, 0.2), 3), source=source)
    if kind == "load":
        n = rng.choice([4, 8, 16])
        return dict(kind=kind, prec=prec, L=_draw_lattice(rng, 4096, 8_000_000 // n), n=n, ru=ru, rn=rn, source=source)
    n = rng.randint(1, 16)
    return dict(kind="cdot", prec="f64", L=_draw_lattice(rng, 4096, 8_000_000 // n), n=n, source=source)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ext(text):
    return tuple(int(a) for a in text.split(","))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _site_signs(L, hop):
    """Staggered phase times the antiperiodic t boundary of a hop, shaped (4, Lt, Lz, Ly, Lx)."""
    x, y, z, t = (torch.arange(a, device="cuda") for a in L)
    x, y, z, t = x.view(1, 1, 1, -1), y.view(1, 1, -1, 1), z.view(1, -1, 1, 1), t.view(-1, 1, 1, 1)
    zero = torch.zeros(L[::-1], dtype=torch.int64, device="cuda")
    odd = torch.stack([zero, zero + x, zero + x + y, zero + x + y + z + (t + hop >= L[3]).long()])
    return 1.0 - 2.0 * (odd & 1).double()


def _haar(gen, count, special):
    """Haar-random U(3) (or SU(3)) matrices: Gram-Schmidt on the columns of complex normal ones."""
    m = torch.randn(count, 3, 3, dtype=torch.complex128, device="cuda", generator=gen)
    cols = []
    for j in range(3):
        c = m[:, :, j]
        for q in cols:
            c = c - q * (q.conj() * c).sum(1, keepdim=True)
        cols.append(c / torch.linalg.vector_norm(c, dim=1, keepdim=True))
    if special:
        a, b, c = cols
        det = (a * torch.linalg.cross(b, c, dim=1)).sum(1, keepdim=True)
        root = torch.polar(torch.ones_like(det.real), -det.angle() / 3.0)
        cols = [v * root for v in cols]
    return torch.stack(cols, dim=2)


def _links(L, gen):
    """Fat links 0.9 x phase x SU(3) and Naik links -1/24 x phase x U(3)."""
    shape = (4,) + tuple(L[::-1]) + (3, 3)
    count = 4 * math.prod(L)
    U = _haar(gen, count, True).view(shape).mul_((FAT * _site_signs(L, 1))[..., None, None])
    N = _haar(gen, count, False).view(shape).mul_((NAIK * _site_signs(L, 3))[..., None, None])
    return U, N


def _vectors(n, sites, source, gen):
    shape = (n, sites, 3)
    if source == "z2":
        s = torch.randint(0, 2, shape + (2,), device="cuda", generator=gen).double().mul_(2.0).sub_(1.0)
        return torch.view_as_complex(s) / math.sqrt(2.0)
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=gen)


def _storage(v, prec):
    """Vectors in the element type of a storage precision, one row per rhs."""
    if prec == "f16":
        return torch.view_as_real(v).to(torch.float16).contiguous()
    return v.to(torch.complex64 if prec == "f32" else torch.complex128).contiguous()


def _rows(t):
    return [t[k] for k in range(t.shape[0])]


def _bundle_buffer(prec, n, vh):
    return torch.empty(n // CHUNK[prec], 3, vh, 2 * CHUNK[prec], device="cuda",
                       dtype=torch.float32 if prec == "f32" else torch.float16)


def _sites(case, L):
    """Sites of the case's vectors: the full lattice or one parity."""
    v = math.prod(L)
    return v if case["kind"] in ("apply", "grad", "cdot") else v // 2


def _load(case, L, U, N):
    return H.hisq_gauge_load(L, U, N, prec=PRECS[case["prec"]], recon_U=case["ru"], recon_N=case["rn"])


def _inputs(case, seed, which=""):
    """Links and source vectors of a case (of its field ``which``), from the seed alone."""
    L, n = _ext(case["L" + which]), case["n" + which]
    gen = _generator(1000003 * int(seed) + int(which or 1))
    U, N = _links(L, gen) if case["kind"] != "cdot" else (None, None)
    return L, U, N, _vectors(n, _sites(case, L), case["source"], gen), gen


def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    if kind == "batched":
        problems = []
        for which in ("", "2", "3"):
            L, U, N, b, _ = _inputs(case, seed, which)
            x = torch.zeros_like(b)
            problems.append(dict(g=_load(case, L, U, N), mass=case["mass"], mu=0.0, b=_rows(b), x=_rows(x), tol=1e-10,
                                 whole=x))
        return dict(case=case, problems=problems,
                    params=H.cg_params(inner_prec=PRECS[prec], reliable_every=case["every"]))
    L, U, N, v, gen = _inputs(case, seed)
    s = dict(case=case, L=L, v=v)
    if kind == "cg":
        s.update(g=_load(case, L, U, N), b=_rows(v), x=torch.zeros_like(v),
                 params=H.cg_params(inner_prec=PRECS[prec], reliable_every=case["every"]))
    elif kind == "grad":
        s.update(U=U.requires_grad_(), N=N.requires_grad_(), b=v.clone().requires_grad_(),
                 mass=torch.tensor(case["mass"], dtype=torch.float64, requires_grad=True),
                 mu=torch.tensor(case["mu"], dtype=torch.float64, requires_grad=True))
    elif kind == "dslash" and case["layout"] == "bundle":
        s.update(g=_load(case, L, U, N), vb=_bundle_buffer(prec, case["n"], v.shape[1]),
                 w=_bundle_buffer(prec, case["n"], v.shape[1]))
        H.hisq_bundle_pack(s["g"], _rows(v), PRECS[prec], s["vb"])
    elif kind in ("dslash", "mdagm", "apply"):
        if case.get("layout") == "soa":
            v = v.transpose(1, 2).contiguous()
        u = _storage(v, prec)
        s.update(g=_load(case, L, U, N), u=u, w=torch.empty_like(u))
    elif kind == "load":
        s.update(U=U, N=N, vb=_bundle_buffer(prec, case["n"], v.shape[1]), w=_bundle_buffer(prec, case["n"], v.shape[1]))
    elif kind == "cdot":
        U, N = _links((4, 4, 4, 4), gen)
        s.update(g=H.hisq_gauge_load((4, 4, 4, 4), U, N, prec=H.HISQ_F64),
                 b=v + 0.5 * _vectors(case["n"], v.shape[1], "gauss", gen))
    return s


def run(s):
    case = s["case"]
    kind, prec = case["kind"], PRECS[case["prec"]]
    if kind == "cg":
        H.hisq_cg_solve(s["g"], case["mass"], 0.0, s["b"], _rows(s["x"]), 1e-10, s["params"])
        return s["x"]
    if kind == "batched":
        H.hisq_cg_solve_batched(s["problems"], s["params"])
        return [p["whole"] for p in s["problems"]]
    if kind == "grad":
        x = A.hisq_solve(s["U"], s["N"], s["mass"], s["mu"], s["b"], 1e-12)
        loss = (s["v"].conj() * x).real.sum()
        g = torch.autograd.grad(loss, (s["U"], s["N"], s["mass"], s["mu"], s["b"]))
        return dict(x=x.detach(), dU=g[0], dN=g[1], dmass=g[2], dmu=g[3], db=g[4])
    if kind == "dslash" and case["layout"] == "bundle":
        H.hisq_dslash_ex(s["g"], case["mu"], s["vb"], s["w"], case["parity"], prec, H.HISQ_BUNDLE, n=case["n"])
    elif kind == "dslash" and case["layout"] == "aos" and case["mu"] == 0.0:
        H.hisq_dslash(s["g"], _rows(s["u"]), _rows(s["w"]), case["parity"], prec)
    elif kind == "dslash":
        H.hisq_dslash_ex(s["g"], case["mu"], _rows(s["u"]), _rows(s["w"]), case["parity"], prec,
                         H.HISQ_SOA if case["layout"] == "soa" else H.HISQ_AOS)
    elif kind == "mdagm":
        H.hisq_mdagm(s["g"], case["mass"], _rows(s["u"]), _rows(s["w"]), prec)
    elif kind == "apply":
        H.hisq_apply_m(s["g"], case["mass"], case["mu"], OPS[case["op"]], _rows(s["u"]), _rows(s["w"]), prec)
    elif kind == "load":
        with _load(case, s["L"], s["U"], s["N"]) as g:
            H.hisq_bundle_pack(g, _rows(s["v"]), prec, s["vb"])
            H.hisq_dslash_ex(g, 0.0, s["vb"], s["w"], 1, prec, H.HISQ_BUNDLE, n=case["n"])
    elif kind == "cdot":
        return np.array(H.hisq_cdot(s["g"], _rows(s["v"]), _rows(s["b"])))
    return s["w"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _dslash_work(vh, n, ru, rn, prec):
    """One Dslash on one parity: every link once, every vector in and out once."""
    r = REAL_BYTES[prec]
    return vh * (8 * (ru + rn) * r + 12 * n * r), FLOPS * n * vh


def _iterations(mass, decades=10):
    """CG iterations of the even-odd system on these links: about 3 / m per decade of the residual."""
    return 3.0 * decades / mass


def work(case):
    kind = case["kind"]
    if kind == "batched":
        parts = [work(dict(case, kind="cg", L=case["L" + w], n=case["n" + w])) for w in ("", "2", "3")]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    L, n, prec = _ext(case["L"]), case["n"], case["prec"]
    vh = math.prod(L) // 2
    if kind == "cdot":
        return {"bytes": 2 * n * 3 * 2 * vh * 16, "flops": 8 * n * 3 * 2 * vh}
    db, df = _dslash_work(vh, n, case["ru"], case["rn"], prec)
    vec = n * vh * 6 * REAL_BYTES[prec]
    links64 = 2 * 4 * 2 * vh * 144                      # both canonical link fields
    if kind == "dslash":
        return {"bytes": db, "flops": df}
    if kind == "mdagm":
        return {"bytes": 2 * db + vec, "flops": 2 * df + 12 * n * vh}
    if kind == "apply":
        return {"bytes": 2 * db + 2 * vec, "flops": 2 * df + 24 * n * vh}
    if kind == "load":
        packed = links64 + 2 * vh * 4 * (case["ru"] + case["rn"]) * REAL_BYTES[prec]   # the FP64 copy and the storage copy
        return {"bytes": links64 + packed + n * vh * 96 + vec + db, "flops": df}
    if kind == "cg":
        it = _iterations(case["mass"])
        return {"bytes": it * (2 * db + 7 * vec), "flops": it * (2 * df + 60 * n * vh)}
    # grad: two full-lattice solves to 1e-12, then the force on every link
    it = 2 * _iterations(case["mass"], 12)
    return {"bytes": it * (4 * db + 14 * vec) + 6 * links64, "flops": it * (4 * df + 120 * n * vh) + 2 * 8 * vh * n * 288}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------

class _Field:
    """D(mu) of Eq. 3 on full-lattice vectors (n, Lt, Lz, Ly, Lx, 3), by array shifts."""

    def __init__(self, L, U, N):
        self.L, self.U, self.N = L, U, N
        x, y, z, t = (torch.arange(a, device="cuda") for a in L)
        self.parity = ((t.view(-1, 1, 1, 1) + z.view(1, -1, 1, 1) + y.view(1, 1, -1, 1) + x.view(1, 1, 1, -1)) & 1).reshape(-1)
        self.order = [torch.nonzero(self.parity == p).view(-1) for p in (0, 1)]

    @staticmethod
    def _mul(m, v):
        return (m * v.unsqueeze(-2)).sum(-1)

    def hops(self, v, factors, directions=range(4)):
        """Sum over the hops, temporal ones with factors (forward, backward) for one and three steps."""
        out = torch.zeros_like(v)
        for mu in directions:
            dim = 4 - mu
            for links, hop, f in ((self.U, 1, factors[0]), (self.N, 3, factors[1])):
                ff, fb = f if mu == 3 else (1.0, 1.0)
                m = links[mu]
                for k in range(v.shape[0]):
                    out[k] += ff * self._mul(m, torch.roll(v[k], -hop, dim - 1))
                    out[k] -= fb * torch.roll(self._mul(m.mH, v[k]), hop, dim - 1)
        return out

    def D(self, v, mu=0.0):
        return self.hops(v, ((math.exp(mu), math.exp(-mu)), (math.exp(3 * mu), math.exp(-3 * mu))))

    def dD(self, v, mu, k):
        """k-th derivative of D(mu) in mu."""
        return self.hops(v, ((math.exp(mu), (-1.0) ** k * math.exp(-mu)),
                             (3.0 ** k * math.exp(3 * mu), (-3.0) ** k * math.exp(-3 * mu))), (3,))

    def spread(self, v, p):
        """Vectors on one parity (n, V_h, 3) as full-lattice ones."""
        out = torch.zeros((v.shape[0], math.prod(self.L), 3), dtype=v.dtype, device=v.device)
        out[:, self.order[p]] = v
        return out.view((v.shape[0],) + tuple(self.L[::-1]) + (3,))

    def take(self, v, p):
        return v.reshape(v.shape[0], -1, 3)[:, self.order[p]]

    def unblock(self, v):
        """Parity-blocked vectors (n, 2 V_h, 3) as full-lattice ones."""
        vh = v.shape[1] // 2
        return self.spread(v[:, :vh], 0) + self.spread(v[:, vh:], 1)

    def block(self, v):
        return torch.cat([self.take(v, 0), self.take(v, 1)], dim=1)

    def M(self, v, mass, mu, dagger=False):
        return 2.0 * mass * v - self.D(v, -mu) if dagger else 2.0 * mass * v + self.D(v, mu)


def _cg(apply, b, tol):
    """Textbook CG with its own coefficients per vector, to a residual of tol."""
    def dot(p, q):
        return (p.conj() * q).real.flatten(1).sum(1)

    def by(c, v):
        return c.view((-1,) + (1,) * (v.dim() - 1)) * v

    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = dot(r, r)
    stop = tol * tol * rr
    for it in range(20000):
        q = apply(p)
        alpha = rr / dot(p, q)
        x += by(alpha, p)
        r -= by(alpha, q)
        new = dot(r, r)
        if it % 10 == 0 and bool((new <= stop).all()):
            break
        p = r + by(new / rr, p)
        rr = new
    return x


def _bundle_of(v, prec):
    """(n, V_h, 3) complex vectors in the bundle layout."""
    w = CHUNK[prec]
    n, vh, _ = v.shape
    r = torch.view_as_real(v).view(n // w, w, vh, 3, 2)
    return r.permute(0, 3, 2, 4, 1).reshape(n // w, 3, vh, 2 * w).contiguous()


def _force(f, mu, hop, a, b):
    """F_hop(a, b) summed over the vectors, canonical link layout."""
    out = torch.zeros_like(f.U)
    for d in range(4):
        ff, fb = (math.exp(hop * mu), math.exp(-hop * mu)) if d == 3 else (1.0, 1.0)
        for k in range(a.shape[0]):
            sa, sb = (torch.roll(v[k], -hop, 3 - d) for v in (a, b))
            out[d] += ff * a[k][..., :, None] * sb[..., None, :].conj() - fb * b[k][..., :, None] * sa[..., None, :].conj()
    return out


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "batched":
        return None
    # plain torch moves tens of KB an iteration for each site and vector: the larger solves would take minutes
    if kind in ("cg", "grad") and _iterations(case["mass"]) * math.prod(_ext(case["L"])) * n > 4.0e8:
        return None
    L, U, N, v, gen = _inputs(case, seed)
    if kind == "cdot":
        _links((4, 4, 4, 4), gen)
        b = v + 0.5 * _vectors(n, v.shape[1], "gauss", gen)
        return (v.conj() * b).flatten(1).sum(1).cpu().numpy()
    f = _Field(L, U, N)
    if kind in ("dslash", "load"):
        p = case.get("parity", 1)
        w = f.take(f.D(f.spread(v, 1 - p), case.get("mu", 0.0)), p)
        layout = case.get("layout", "bundle")
        if layout == "bundle":
            return _bundle_of(w, case["prec"])
        w = w.transpose(1, 2).contiguous() if layout == "soa" else w
        return torch.view_as_real(w.contiguous()) if case["prec"] == "f16" else w
    if kind == "mdagm":
        w = 4.0 * case["mass"] ** 2 * v - f.take(f.D(f.D(f.spread(v, 0))), 0)
        return torch.view_as_real(w.contiguous()) if case["prec"] == "f16" else w
    if kind == "apply":
        u = f.unblock(v)
        if case["op"] in ("M", "Mdag"):
            w = f.M(u, case["mass"], case["mu"], case["op"] == "Mdag")
        else:
            w = f.dD(u, case["mu"], 1 if case["op"] == "dM" else 2)
        w = f.block(w)
        return torch.view_as_real(w.contiguous()) if case["prec"] == "f16" else w
    m = case["mass"]
    if kind == "cg":
        return f.take(_cg(lambda q: 4.0 * m * m * q - f.D(f.D(q)), f.spread(v, 0), 1e-13), 0)
    # grad of sum Re eta^dag x: lambda solves the adjoint system with eta, which is also the source
    mu, b = case["mu"], f.unblock(v)
    x = _cg(lambda q: f.M(f.M(q, m, mu), m, mu, True), b, 1e-14)
    y = f.M(x, m, mu)
    dot = lambda p, q: (p.conj() * q).real.sum()  # noqa: E731
    dy = f.dD(x, mu, 1)
    return dict(x=f.block(x), dU=-2.0 * _force(f, mu, 1, y, x), dN=-2.0 * _force(f, mu, 3, y, x),
                dmass=-4.0 * dot(y, x).cpu(), dmu=-2.0 * dot(y, dy).cpu(), db=f.block(x))

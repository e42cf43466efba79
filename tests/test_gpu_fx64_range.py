"""FP64 operators on links and vectors whose products differ widely in size.

Every output real is held to the bound of 96 FP64 fused multiply-adds on its
own products: |error| <= 96 x 2^-53 x sum |m| |v| over the products of that
real (4 more units where a temporal factor scales the link, 2 more for the
mass term). The reference sums in long double. A sum that keeps its bits
relative to anything larger than its own products (a neighbour behind a zero
link, another colour, another direction's links) breaks it.
"""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -53
LD, CLD = np.longdouble, np.clongdouble


def reals(z):
    return np.stack([z.real, z.imag], axis=-1)


def hops(U, N, factors, directions=range(4)):
    """(direction, steps, links as they multiply the neighbour, factor) of Eq. 3."""
    for mu in directions:
        for links, d in ((U, 1), (N, 3)):
            f, b = factors[d] if mu == 3 else (1.0, 1.0)
            yield mu, d, links[mu], f
            back = np.conj(np.swapaxes(np.roll(links[mu], d, axis=3 - mu), -1, -2))
            yield mu, -d, -back, b


def exact(U, N, v, L, parity, factors, directions=range(4)):
    """Long-double D v on one parity, (n, V_h, 3, 2), and the sums of |products| of each real."""
    full = np.zeros((v.shape[0],) + O.grid_shape(L) + (3,), dtype=CLD)
    full[:, O.parity_mask(L, 1 - parity)] = v
    out = np.zeros(full.shape, dtype=CLD)
    size = np.zeros(full.shape + (2,), dtype=LD)
    for mu, d, m, f in hops(U, N, factors, directions):
        w = np.roll(full, -d, axis=4 - mu)
        m = m.astype(CLD) * LD(f)
        out += np.einsum("tzyxij,ntzyxj->ntzyxi", m, w)
        a, b, p, q = abs(m.real), abs(m.imag), abs(w.real), abs(w.imag)
        mul = lambda s, t: np.einsum("tzyxij,ntzyxj->ntzyxi", s, t)  # noqa: E731
        size[..., 0] += mul(a, p) + mul(b, q)
        size[..., 1] += mul(a, q) + mul(b, p)
    mask = O.parity_mask(L, parity)
    return reals(out[:, mask]), size[:, mask]


def exp_factors(mu):
    return {1: (np.exp(mu), np.exp(-mu)), 3: (np.exp(3.0 * mu), np.exp(-3.0 * mu))}


def within(got, ref, size, units):
    err = abs(reals(got).astype(LD) - ref)
    assert np.isfinite(err.astype(float)).all()
    # below the smallest normal number a product is rounded to a subnormal
    worst = (err / (units * UNIT * size + 96 * LD(2.0) ** -1074)).max()
    assert worst <= 1.0, f"error is {float(worst):.3g} times the bound"


def load(H, L, U, N, prec=0, **kw):
    import torch
    return H.hisq_gauge_load(L, torch.from_numpy(U).cuda(), torch.from_numpy(N).cuda(), prec=prec, **kw)


def dslash(H, g, v, parity, mu=0.0, rpt=0, layout=0):
    import torch
    H.hisq_set_dslash_mapping(g, rpt)
    vd = [torch.from_numpy(np.ascontiguousarray(x.T if layout == H.HISQ_SOA else x)).cuda() for x in v]
    wd = [torch.full_like(t, float("nan")) for t in vd]
    H.hisq_dslash_ex(g, mu, vd, wd, parity, H.HISQ_F64, layout)
    torch.cuda.synchronize()
    w = [t.cpu().numpy() for t in wd]
    return np.stack([x.T if layout == H.HISQ_SOA else x for x in w])


def structured(kind, L, n, seed):
    """Links and full-lattice vectors whose sums need bits far below the largest neighbour."""
    rng = np.random.default_rng(seed)
    U, N = gen.hisq_links(L, seed=seed)
    V = int(np.prod(L))
    v = rng.standard_normal((n, V, 3)) + 1j * rng.standard_normal((n, V, 3))
    grid = np.zeros(O.grid_shape(L), dtype=int) + np.arange(L[3]).reshape(-1, 1, 1, 1)
    t = np.concatenate([grid[O.parity_mask(L, p)] for p in (0, 1)])
    name, _, arg = kind.partition(" ")
    s = float(arg) if arg else 1.0
    if name == "no-naik":                 # an empty block beside small links
        U *= s
        N[:] = 0.0
    elif name == "no-fat":
        U[:] = 0.0
    elif name == "no-direction":
        U[2] = N[2] = 0.0
        U *= s
    elif name == "cut":                   # open temporal boundary, vectors of another size behind it
        U[3, -1] = 0.0
        N[3, -3:] = 0.0
        v[:, t >= L[3] // 2] *= s
        U[3, L[3] // 2 - 1] = 0.0
        N[3, L[3] // 2 - 3:L[3] // 2] = 0.0
    elif name == "colours":               # abelian links, colours of different size
        for links in (U, N):
            size = np.abs(links).max()
            links[:] = size * np.eye(3) * np.exp(1j * rng.uniform(0, 6.28, links.shape[:-1]))[..., None]
        v[..., 0] *= s
    elif name == "off-diagonal":          # nearly abelian: small entries carry an output alone
        for links in (U, N):
            mix = links * 1e-10
            size = np.abs(links).max()
            links[:] = size * np.eye(3) * np.exp(1j * rng.uniform(0, 6.28, links.shape[:-1]))[..., None] + mix
        v[..., 1:] = 0.0
    elif name == "patch":                 # the same on a quarter of the time slices, cut off from the others
        quarter = L[3] // 4
        for links, d in ((U, 1), (N, 3)):
            size = np.abs(links).max()
            part = links[:, :quarter]
            part[:] = size * np.eye(3) * np.exp(1j * rng.uniform(0, 6.28, part.shape[:-1]))[..., None]
            links[3, max(quarter - d, 0):quarter] = 0.0
            links[3, -d:] = 0.0
        v[..., 0] *= s
    elif name == "real":                  # real links, imaginary parts of another size
        U, N = U.real + 0j, N.real + 0j
        v = v.real + 1j * s * v.imag
    elif name == "nearly-real":
        U, N = U.real + 1e-11j * U.imag, N.real + 1e-11j * N.imag
        v = v.real + 0j
    elif name == "uneven":                # links of one direction from 1 to s
        for links in (U, N):
            links *= np.exp(rng.uniform(0, np.log(s), links.shape[:-2]))[..., None, None]
    elif name == "point":                 # one site, one colour
        v[:] = 0.0
        v[np.arange(n), rng.integers(0, V, n), np.arange(n) % 3] = 1.0
    elif name == "decay":                 # sizes falling by s from one time slice to the next
        v *= (s ** t)[:, None]
    else:
        assert name == "haar"
    return U, N, v


KINDS = ["haar", "no-naik", "no-naik 1e-2", "no-naik 1e-8", "no-naik 1e-17", "no-fat", "no-direction 1e-9", "cut 1e3",
         "cut 1e18", "colours 1e-3", "colours 1e-8", "colours 1e-14", "patch 1e-2", "patch 1e-9", "off-diagonal", "real 1e-9", "nearly-real",
         "uneven 3", "uneven 15", "point", "decay 0.1", "decay 1e-6"]


SMALL, ONE, TWO, FOUR = ((4, 6, 8, 10), 2, 1), ((8, 8, 8, 10), 8, 1), ((8, 12, 10, 14), 8, 2), ((4, 6, 10, 8), 4, 4)


# four lanes a site (the small lattice) and one, one, two and four rhs a thread,
# ragged last blocks; the first and last rhs are compared
@pytest.mark.parametrize("kind,shape", [(k, s) for s in (SMALL, ONE, FOUR) for k in KINDS] +
                         [(k, TWO) for k in ("no-naik 1e-8", "cut 1e18", "patch 1e-9", "point")])
def test_dslash_keeps_the_bits_of_every_real(gpu_lib, kind, shape):
    L, n, rpt = shape
    U, N, v = structured(kind, L, n, seed=31)
    half = v.shape[1] // 2
    some = [0, n - 1]
    g = load(gpu_lib, L, U, N)
    try:
        for parity, layout in ((0, 0), (1, 1)):
            w = v[:, half:] if parity == 0 else v[:, :half]
            ref, size = exact(U, N, w[some], L, parity, exp_factors(0.0))
            within(dslash(gpu_lib, g, w, parity, 0.0, rpt, layout)[some], ref, size, 96)
    finally:
        gpu_lib.hisq_gauge_free(g)


@pytest.mark.parametrize("kind", KINDS)
def test_full_lattice_operators_keep_the_bits_of_every_real(gpu_lib, kind):
    import torch
    H = gpu_lib
    L, n, mass, mu = (4, 6, 8, 6), 2, 0.07, 0.2
    U, N, v = structured(kind, L, n, seed=32)
    half = v.shape[1] // 2
    vd = [torch.from_numpy(x).cuda() for x in v]
    e = exp_factors(mu)
    derivative = {d: (d * e[d][0], -d * e[d][1]) for d in (1, 3)}
    adjoint = {d: e[d][::-1] for d in (1, 3)}
    g = load(H, L, U, N)
    try:
        for op, sign, f, m, directions in ((H.HISQ_OP_M, 1, e, mass, range(4)), (H.HISQ_OP_MDAG, -1, adjoint, mass, range(4)),
                                           (H.HISQ_OP_DM_DMU, 1, derivative, 0.0, (3,))):
            wd = [torch.full_like(t, float("nan")) for t in vd]
            H.hisq_apply_m(g, mass, mu, op, vd, wd, H.HISQ_F64)
            torch.cuda.synchronize()
            got = np.stack([t.cpu().numpy() for t in wd])
            for p in (0, 1):
                mine, other = (v[:, p * half:(p + 1) * half], v[:, (1 - p) * half:(2 - p) * half])
                ref, size = exact(U, N, other, L, p, f, directions)
                ref = sign * ref + 2 * LD(m) * reals(mine)
                size = size + 2 * m * abs(reals(mine))
                within(got[:, p * half:(p + 1) * half], ref, size, 102)
    finally:
        H.hisq_gauge_free(g)


@pytest.mark.parametrize("mu", [-60.0, -30.0, -16.0, -5.0, 5.0, 12.0, 16.0, 20.0, 30.0, 60.0])
def test_large_temporal_factors(gpu_lib, mu):
    """Zero stays zero, non-finite neighbours are seen behind any factor, the rest keeps its bits."""
    L, n = (4, 6, 8, 10), 2
    U, N, v = structured("haar", L, n, seed=33)
    v = np.ascontiguousarray(v[:, v.shape[1] // 2:])
    g = load(gpu_lib, L, U, N)
    try:
        ref, size = exact(U, N, v, L, 0, exp_factors(mu))
        within(dslash(gpu_lib, g, v, 0, mu), ref, size, 102)
        assert not dslash(gpu_lib, g, 0.0 * v, 0, mu).any()
        for bad in (np.inf, -np.inf, np.nan):
            w = v.copy()
            w[n - 1, 17, 1] = bad
            with np.errstate(invalid="ignore"):
                want = np.isfinite(O.dslash_parity(U, N, w, L, 0, mu))
            got = dslash(gpu_lib, g, w, 0, mu)
            assert (np.isfinite(got) == want).all() and not want.all()
    finally:
        gpu_lib.hisq_gauge_free(g)


def test_small_and_large_links(gpu_lib):
    """Fields of size 2^-150 to 2^150, and zero vectors on them."""
    L, n = (4, 6, 8, 10), 2
    for scale in (-150, -70, 40, 62, 90, 120, 150):
        U, N, v = structured("haar", L, n, seed=34)
        U, N, v = 2.0 ** scale * U, 2.0 ** scale * N, np.ascontiguousarray(v[:, v.shape[1] // 2:])
        g = load(gpu_lib, L, U, N)
        try:
            ref, size = exact(U, N, v, L, 0, exp_factors(0.0))
            within(dslash(gpu_lib, g, v, 0), ref, size, 96)
            assert not dslash(gpu_lib, g, 0.0 * v, 0).any()
        finally:
            gpu_lib.hisq_gauge_free(g)

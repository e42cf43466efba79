"""The FP64 Dslash's fixed-point sums against the oracle where they can go wrong.

Every sum carries 55 to 56 bits below the largest neighbour component of its
site: 96 products rounded at no more than 3 x 2^-56 of the largest product
stay within 96 x 3 x 2^-56 = 4e-15 of it, and the output of a site of Haar
links is no smaller than a few per cent of it. Bound used per site: 1e-13.
"""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O
from conftest import from_dev, rel_l2, to_dev

pytestmark = pytest.mark.gpu


def dslash(H, L, U, N, v, parity, mu=0.0, rpt=0, layout=0):
    import torch
    g = H.hisq_gauge_load(L, torch.from_numpy(U).cuda(), torch.from_numpy(N).cuda(), prec=H.HISQ_F64)
    try:
        if rpt:
            H.hisq_set_dslash_mapping(g, rpt)
        vd = [to_dev(v[k], 0) for k in range(len(v))]
        if layout == H.HISQ_SOA:
            vd = [t.t().contiguous() for t in vd]
        wd = [torch.full_like(t, float("nan")) for t in vd]
        H.hisq_dslash_ex(g, mu, vd, wd, parity, H.HISQ_F64, layout)
        torch.cuda.synchronize()
        if layout == H.HISQ_SOA:
            wd = [t.t().contiguous() for t in wd]
        return np.stack([from_dev(t) for t in wd])
    finally:
        H.hisq_gauge_free(g)


def site_error(got, ref):
    big = np.abs(ref).max()   # keeps the squares in range
    return (np.linalg.norm((got - ref) / big, axis=-1) / np.linalg.norm(ref / big, axis=-1)).max()


# one lane per direction (few sites) and one lane per site, one, two and four rhs per thread, a ragged last block
@pytest.mark.parametrize("L,n,rpt", [((4, 4, 4, 4), 1, 1), ((4, 6, 10, 8), 3, 1), ((4, 6, 10, 8), 4, 2), ((4, 6, 8, 10), 8, 4),
                                     ((8, 12, 10, 14), 14, 2), ((16, 12, 10, 14), 8, 1), ((16, 12, 10, 14), 6, 2)])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("mu", [0.0, -0.3])
def test_sites_of_very_different_size(gpu_lib, L, n, rpt, layout, mu):
    U, N = gen.hisq_links(L, seed=5)
    rng = np.random.default_rng(6)
    v = gen.gaussian_source(L, n, seed=7)
    v *= np.exp2(rng.integers(-60, 61, size=v.shape[:2]))[..., None]   # neighbours up to 2^120 apart
    v[:, rng.random(v.shape[1]) < 0.1] = 0.0
    ref = O.dslash_parity(U, N, v, L, 1, mu)
    got = dslash(gpu_lib, L, U, N, v, 1, mu, rpt, layout)
    assert site_error(got, ref) < 1e-13


@pytest.mark.parametrize("n,rpt", [(1, 1), (2, 2)])
def test_zero_extreme_and_nonfinite_vectors(gpu_lib, n, rpt):
    L = (4, 6, 8, 10)
    U, N = gen.hisq_links(L, seed=5)
    v = gen.gaussian_source(L, n, seed=8)
    ref = O.dslash_parity(U, N, v, L, 0)
    assert not dslash(gpu_lib, L, U, N, 0.0 * v, 0, rpt=rpt).any()
    assert not dslash(gpu_lib, L, U, N, -0.0 * v, 0, rpt=rpt).any()
    for scale in (1e-290, 1e-200, 1e200, 1e290):
        assert site_error(dslash(gpu_lib, L, U, N, scale * v, 0, rpt=rpt), scale * ref) < 1e-13
    for bad in (np.inf, -np.inf, np.nan):
        w = v.copy()
        w[n - 1, 17, 1] = bad
        with np.errstate(invalid="ignore"):
            want = np.isfinite(O.dslash_parity(U, N, w, L, 0))
        got = dslash(gpu_lib, L, U, N, w, 0, rpt=rpt)
        assert (np.isfinite(got) == want).all() and not want.all()
        assert rel_l2(got[want], ref[want]) < 1e-13


@pytest.mark.parametrize("mu", [0.0, 0.2, 100.0, -150.0])
def test_links_of_different_size_and_large_factors(gpu_lib, mu):
    """Directions of different size stay in fixed point, links of one direction 1e6 apart do not."""
    L = (4, 6, 8, 6)
    U, N = gen.hisq_links(L, seed=9)
    v = gen.gaussian_source(L, 2, seed=10)
    U[1] *= 1e-5
    N[2] *= 300.0
    U[0, 0] = 0.0
    V = U.copy()
    V[2, ::2] *= 1e-6
    for links in (U, V):
        ref = O.dslash_parity(links, N, v, L, 0, mu)
        assert site_error(dslash(gpu_lib, L, links, N, v, 0, mu), ref) < 1e-13


# both parities in one launch: every operator, in place of two launches; bound as above
@pytest.mark.parametrize("L,n", [((4, 4, 4, 6), 1), ((4, 6, 10, 8), 3), ((12, 12, 10, 14), 4)])
def test_full_lattice_operators_take_both_parities(gpu_lib, L, n):
    import torch
    H = gpu_lib
    U, N = gen.hisq_links(L, seed=11)
    m, mu = 0.07, 0.15
    g = H.hisq_gauge_load(L, torch.from_numpy(U).cuda(), torch.from_numpy(N).cuda(), prec=H.HISQ_F64)
    try:
        rng = np.random.default_rng(12)
        V = int(np.prod(L))
        v = rng.standard_normal((n, V, 3)) + 1j * rng.standard_normal((n, V, 3))
        vd = [torch.from_numpy(v[k]).cuda() for k in range(n)]
        halves = (v[:, :V // 2], v[:, V // 2:])
        for op, sgn, muf, mass in ((H.HISQ_OP_M, 1.0, mu, m), (H.HISQ_OP_MDAG, -1.0, -mu, m)):
            wd = [torch.full_like(t, float("nan")) for t in vd]
            H.hisq_apply_m(g, m, mu, op, vd, wd, H.HISQ_F64)
            torch.cuda.synchronize()
            for p in (0, 1):
                ref = 2 * mass * halves[p] + sgn * O.dslash_parity(U, N, halves[1 - p], L, p, muf)
                got = np.stack([t.cpu().numpy()[p * (V // 2):(p + 1) * (V // 2)] for t in wd])
                assert site_error(got, ref) < 1e-13
    finally:
        H.hisq_gauge_free(g)

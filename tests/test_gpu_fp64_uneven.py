"""FP64 operators and solves on fields that keep to multiply-adds.

One link a thousand times smaller than the others takes a field off the
fixed-point links, so the FP64 multiply-add kernels run: both layouts, every
rhs per thread, all epilogues, the reductions of the solves and of the
reliable updates, and the full-lattice operators with a launch per parity.
"""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O
from conftest import from_dev, rel_l2, to_dev
from test_gpu_cg import oracle_solution, solve
from test_gpu_fx64_range import dslash, exact, exp_factors, load, within

pytestmark = pytest.mark.gpu


def uneven_links(L, seed):
    U, N = gen.hisq_links(L, seed=seed)
    U[0, 1, 2, 3, 1] *= 1e-3
    return U, N


@pytest.mark.parametrize("L,n,rpt", [((4, 6, 8, 10), 3, 1), ((4, 6, 8, 10), 6, 2), ((4, 8, 6, 10), 8, 4), ((4, 6, 8, 10), 4, 0)])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("mu", [0.0, -0.3])
def test_dslash(gpu_lib, L, n, rpt, layout, mu):
    U, N = uneven_links(L, 51)
    v = gen.gaussian_source(L, n, seed=52)
    g = load(gpu_lib, L, U, N)
    try:
        some = [0, n - 1]
        for parity in (0, 1):
            ref, size = exact(U, N, v[some], L, parity, exp_factors(mu))
            within(dslash(gpu_lib, g, v, parity, mu, rpt, layout)[some], ref, size, 102)
    finally:
        gpu_lib.hisq_gauge_free(g)


# tolerances of the same operators on even fields: 1e-13 of the norm
@pytest.mark.parametrize("n", [1, 4])
def test_operators(gpu_lib, n):
    import torch
    H = gpu_lib
    L, m, mu = (4, 6, 8, 10), 0.07, 0.15
    U, N = uneven_links(L, 53)
    rng = np.random.default_rng(54)
    V = int(np.prod(L))
    v = rng.standard_normal((n, V, 3)) + 1j * rng.standard_normal((n, V, 3))
    full = O.to_full(v[:, :V // 2], L, 0) + O.to_full(v[:, V // 2:], L, 1)
    g = load(H, L, U, N)
    try:
        vd = [torch.from_numpy(x).cuda() for x in v]
        for op, ref in ((H.HISQ_OP_M, O.apply_M(U, N, full, m, mu)), (H.HISQ_OP_MDAG, O.apply_Mdag(U, N, full, m, mu)),
                        (H.HISQ_OP_DM_DMU, O.apply_dM_dmu(U, N, full, mu)),
                        (H.HISQ_OP_D2M_DMU2, O.apply_dnM_dmun(U, N, full, mu, 2))):
            wd = [torch.full_like(t, float("nan")) for t in vd]
            H.hisq_apply_m(g, m, mu, op, vd, wd, H.HISQ_F64)
            torch.cuda.synchronize()
            got = np.stack([t.cpu().numpy() for t in wd])
            assert rel_l2(got[:, :V // 2], O.to_half(ref, L, 0)) < 1e-13
            assert rel_l2(got[:, V // 2:], O.to_half(ref, L, 1)) < 1e-13
        b = v[:, :V // 2]
        bd = [to_dev(x, H.HISQ_F64) for x in b]
        wd = [torch.full_like(t, float("nan")) for t in bd]
        H.hisq_mdagm(g, m, bd, wd, H.HISQ_F64)
        torch.cuda.synchronize()
        assert rel_l2(np.stack([from_dev(t) for t in wd]), O.apply_Ae(U, N, b, L, m)) < 1e-13
    finally:
        H.hisq_gauge_free(g)


# prec 0: FP64 inner iterations; 1 and 2: FP64 reliable updates; the solves' own tolerances
@pytest.mark.parametrize("prec,n", [(0, 1), (0, 4), (1, 2), (1, 8), (2, 4)])
def test_even_odd_solve(gpu_lib, prec, n):
    L, m = (4, 6, 4, 6), 0.1
    U, N = uneven_links(L, 55)
    b = gen.z2_source(L, n, seed=56)
    x, st = solve(gpu_lib, L, U, N, b, m, prec=prec, rn=18)
    xo, A = oracle_solution(U, N, L, b, m)
    res = O.true_relative_residual(A, x, b)
    assert np.all(res <= 1e-10)
    assert np.all(np.abs(np.array(st.true_rel_res[:n]) - res) <= 1e-11)
    assert rel_l2(x, xo) <= 1e-8


@pytest.mark.parametrize("prec", [0, 1])
def test_full_lattice_solve(gpu_lib, prec):
    L, m, mu, n = (4, 4, 4, 6), 0.1, 0.1, 2
    U, N = uneven_links((4, 4, 4, 6), 57)
    be, bo = gen.z2_source(L, n, seed=58), gen.z2_source(L, n, seed=59)
    x, st = solve(gpu_lib, L, U, N, np.concatenate([be, bo], axis=1), m, prec=prec, rn=18, mu=mu)
    b = O.to_full(be, L, 0) + O.to_full(bo, L, 1)
    vh = be.shape[1]
    full = O.to_full(x[:, :vh], L, 0) + O.to_full(x[:, vh:], L, 1)
    xo, A = oracle_solution(U, N, L, b, m, mu=mu)
    assert np.all(O.true_relative_residual(A, full, b) <= 1e-10)
    assert rel_l2(full, xo) <= 1e-8

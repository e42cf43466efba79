"""Reductions over more tiles than there are partial-sum slots.

Beyond 16384 tiles a block of a Dslash with a reduction takes several
consecutive ones. 32 x 32 x 32 x 36 sites with 12 rhs make 18432 tiles of 32
sites, in the bundle kernels and in the FP64 kernel of the reliable updates.
"""
import pytest

pytestmark = pytest.mark.gpu


# bound: the residual the solve reports is that of its solution under the FP64
# operator, to the rounding of either (1e-12 of |b|)
@pytest.mark.parametrize("prec", [1, 2])
def test_solve_with_several_tiles_a_block(gpu_lib, prec):
    import torch
    H = gpu_lib
    L, n, m = (32, 32, 32, 36), 12, 0.5
    V = 32 ** 3 * 36
    gen = torch.Generator(device="cuda").manual_seed(61)

    def links():
        q = torch.randn(4 * V, 3, 3, dtype=torch.complex128, device="cuda", generator=gen)
        cols = []
        for j in range(3):
            c = q[:, :, j]
            for e in cols:
                c = c - e * (e.conj() * c).sum(1, keepdim=True)
            cols.append(c / torch.linalg.vector_norm(c, dim=1, keepdim=True))
        return torch.stack(cols, dim=2).view((4,) + L[::-1] + (3, 3))

    U, N = 0.9 * links(), links() / 24
    b = torch.randn(n, V // 2, 3, dtype=torch.complex128, device="cuda", generator=gen)
    x, r = torch.zeros_like(b), torch.empty_like(b)
    with H.hisq_gauge_load(L, U, N, prec=prec, recon_U=18, recon_N=14) as g:
        st = H.hisq_cg_solve(g, m, 0.0, list(b), list(x), 1e-10, H.cg_params(inner_prec=prec))
        H.hisq_mdagm(g, m, list(x), list(r), H.HISQ_F64)
    res = (torch.linalg.vector_norm((r - b).flatten(1), dim=1) / torch.linalg.vector_norm(b.flatten(1), dim=1)).tolist()
    # |D| <= 8 (0.9 + 1/24), so the condition is at most 57 and textbook CG takes sqrt(57) / 2 x ln(2e10) = 90 iterations
    assert max(res) <= 1e-10 and st.total_iters < 180
    assert max(abs(st.true_rel_res[k] - res[k]) for k in range(n)) <= 1e-12

"""R14 loading where the pivot of z = row3_k / conj(row1 x row2)_k can go wrong.

Permutation links leave one nonzero pivot, each of the three in turn; small
links take the pivot search out of FP32 range. Bounds: those of the Dslash in
the storage precision (F32 1e-6, F16 3e-3).
"""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O
from conftest import from_dev, rel_l2, to_dev

pytestmark = pytest.mark.gpu


# small and large links in F32 only: half vectors would leave their range
@pytest.mark.parametrize("prec,tol,kind,scale", [(1, 1e-6, "permutation", 1.0), (2, 3e-3, "permutation", 1.0),
                                                 (1, 1e-6, "haar", 1e-9), (1, 1e-6, "haar", 3e5)])
def test_r14_pivots_and_sizes(gpu_lib, prec, tol, kind, scale):
    import torch
    H = gpu_lib
    L = (4, 6, 8, 6)
    U, N = gen.hisq_links(L, seed=4)
    if kind == "permutation":
        rng = np.random.default_rng(5)
        for links in (U, N):
            flat = links.reshape(-1, 3, 3)
            size = np.linalg.norm(flat[0, 0])
            eye = np.eye(3)
            perms = [eye[list(p)] for p in ((0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 2, 1), (2, 1, 0), (1, 0, 2))]
            flat[:] = size * np.stack([perms[k] for k in rng.integers(0, 6, len(flat))])
            flat *= np.exp(1j * rng.uniform(0, 6, (len(flat), 3, 1)))
    U, N = scale * U, scale * N
    g = H.hisq_gauge_load(L, torch.from_numpy(U).cuda(), torch.from_numpy(N).cuda(), prec=prec, recon_U=14, recon_N=14,
                          recon_tol=1e-10 * max(scale, 1.0))
    try:
        v = gen.gaussian_source(L, 2, seed=6)
        vd = [to_dev(v[k], prec) for k in range(2)]
        wd = [torch.empty_like(t) for t in vd]
        H.hisq_dslash(g, vd, wd, 0, prec)
        torch.cuda.synchronize()
        ref = O.dslash_parity(U, N, np.stack([from_dev(t) for t in vd]), L, 0)
        for k in range(2):
            assert rel_l2(from_dev(wd[k]), ref[k]) < tol
    finally:
        H.hisq_gauge_free(g)

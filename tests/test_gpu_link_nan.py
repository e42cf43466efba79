"""A NaN link in a 16-bit field spoils its own sites only.

The scales of the 16-bit links come from the largest numbers of the field.
Bound: that of the Dslash in 16-bit storage, 3e-3.
"""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O
from conftest import from_dev, rel_l2, to_dev

pytestmark = pytest.mark.gpu


# the element of the link: with R14 the pivot of the third row must not meet the NaN
@pytest.mark.parametrize("recon,row,col", [(18, 0, 0), (18, 2, 1), (14, 0, 0)])
@pytest.mark.parametrize("naik", [0, 1])
def test_one_nan_link_spoils_its_own_sites(gpu_lib, recon, row, col, naik):
    import torch
    H = gpu_lib
    L = (4, 6, 8, 6)
    U, N = gen.hisq_links(L, seed=21)
    bad = [U.copy(), N.copy()]
    bad[naik][1, 2, 3, 4, 1, row, col] = complex(np.nan, 0.1)
    g = H.hisq_gauge_load(L, torch.from_numpy(bad[0]).cuda(), torch.from_numpy(bad[1]).cuda(), prec=H.HISQ_F16,
                          recon_U=recon, recon_N=recon)
    try:
        for parity in (0, 1):
            v = [to_dev(x, H.HISQ_F16) for x in gen.gaussian_source(L, 2, seed=22)]
            w = [torch.empty_like(t) for t in v]
            H.hisq_dslash(g, v, w, parity, H.HISQ_F16)
            torch.cuda.synchronize()
            src = np.stack([from_dev(t) for t in v])
            with np.errstate(invalid="ignore"):
                well = np.isfinite(O.dslash_parity(bad[0], bad[1], src, L, parity)).all(axis=(0, 2))
            assert 0 < (~well).sum() <= 2
            ref = O.dslash_parity(U, N, src, L, parity)
            got = np.stack([from_dev(t) for t in w])
            assert rel_l2(got[:, well], ref[:, well]) < 3e-3
    finally:
        H.hisq_gauge_free(g)

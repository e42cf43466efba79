"""The mapping of FP64 calls on fields with and without fixed-point links."""
import numpy as np
import pytest

import hisq_inputs as gen
from oracle import hisq_oracle as O
from conftest import from_dev, rel_l2, to_dev

pytestmark = pytest.mark.gpu

L = (4, 6, 8, 10)


def fields(seed):
    """Links of one size, and the same with one link off (which keep to multiply-adds)."""
    U, N = gen.hisq_links(L, seed=seed)
    W = U.copy()
    W[0, 1, 2, 3, 1] *= 1e-3
    return (U, N), (W, N)


def test_reported_mapping_is_the_one_that_runs(gpu_lib):
    import torch
    H = gpu_lib
    even, uneven = fields(41)
    for (U, N), mapping in ((even, (2, 3, 0)), (uneven, (2, 2, H.HISQ_MAP_L2_PREFETCH))):
        with H.hisq_gauge_load(L, torch.from_numpy(U).cuda(), torch.from_numpy(N).cuda(), prec=H.HISQ_F64) as g:
            H.hisq_set_dslash_mapping(g, 2, 2, H.HISQ_MAP_L2_PREFETCH)
            assert H.hisq_get_dslash_mapping(g, 4, H.HISQ_F64) == mapping


def test_tuned_mappings_of_one_kind_of_field_stay_with_it(gpu_lib):
    import torch
    H = gpu_lib
    n = 4
    even, uneven = fields(42)
    with H.hisq_gauge_load_tuned(L, torch.from_numpy(even[0]).cuda(), torch.from_numpy(even[1]).cuda(), H.HISQ_F64, n):
        pass
    U, N = (torch.from_numpy(x).cuda() for x in uneven)
    with H.hisq_gauge_load(L, U, N, prec=H.HISQ_F64) as g:
        default = H.hisq_get_dslash_mapping(g, n, H.HISQ_F64)
    with H.hisq_gauge_load_tuned(L, U, N, H.HISQ_F64, n) as g:
        assert H.hisq_get_dslash_mapping(g, n, H.HISQ_F64) == default
        b = gen.gaussian_source(L, n, seed=43)
        v = [to_dev(x, H.HISQ_F64) for x in b]
        w = [torch.empty_like(t) for t in v]
        H.hisq_dslash(g, v, w, 0, H.HISQ_F64)
        torch.cuda.synchronize()
        ref = O.dslash_parity(uneven[0], uneven[1], b, L, 0)
        assert rel_l2(np.stack([from_dev(t) for t in w]), ref) < 1e-14

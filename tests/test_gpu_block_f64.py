"""The coded double kernels (groups of four 9-node blocks, lines by parity
class): block counts of every remainder modulo four, every level count, ROI
tiers per block of a group, coefficients at the range check's edge, and fields
so large that sums of four values overflow."""
import numpy as np
import pytest
import torch

import fields
import oracle
from _util import check_stream_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(9, 9, 9), (9, 10, 9), (9, 9, 27), (18, 9, 19), (20, 19, 21)])
@pytest.mark.parametrize("K", [1, 2, 3])
def test_groups_of_nine_node_blocks(shape, K):
    import paper_2609_00205_gb300 as bm

    u = fields.power_law_grf(shape, exponent=-2.0, seed=sum(shape), dtype=torch.float64).numpy()
    for tol in (1e-2, 1e-6, 1e-10):
        s = bm.compress(torch.from_numpy(u).to("cuda"), tol, block=9, levels=K, global_levels=1).cpu().numpy()
        check_stream_parity(bm, u, s, tol, "rel", 9, K, 1, label=f"f64_groups_{shape}_{K}")


@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_seventeen_node_blocks(K):
    import paper_2609_00205_gb300 as bm

    u = fields.power_law_grf((20, 35, 18), exponent=-2.0, seed=K, dtype=torch.float64).numpy()
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-5, block=17, levels=K, global_levels=1).cpu().numpy()
    check_stream_parity(bm, u, s, 1e-5, "rel", 17, K, 1, label=f"f64_b17_{K}")


def test_roi_tiers_within_a_group():
    import paper_2609_00205_gb300 as bm

    shape = (20, 19, 21)
    u = fields.power_law_grf(shape, exponent=-2.0, seed=3, dtype=torch.float64).numpy()
    nb = int(np.prod([-(-n // 9) for n in shape]))
    roi = np.array([1e-3, 1e-7, 1e-5, 1e-2])[np.arange(nb) * 7 % 4]
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-2, roi=roi, block=9, levels=2, global_levels=1).cpu().numpy()
    check_stream_parity(bm, u, s, 1e-2, "rel", 9, 2, 1, roi=roi, label="f64_groups_roi")


@pytest.mark.parametrize("B,K", [(9, 2), (17, 2)])
def test_sums_that_overflow_give_the_oracles_raw_copy(B, K):
    import paper_2609_00205_gb300 as bm

    u = fields.power_law_grf((20, 19, 21), exponent=-2.0, seed=5, dtype=torch.float64).numpy()
    u = u / np.abs(u).max() * 1.7e308
    so = oracle.compress(u, 1e-3, rel=True, B=B, K=K, M=1)
    assert oracle.stream_header(so)["raw"]
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-3, block=B, levels=K, global_levels=1).cpu().numpy()
    np.testing.assert_array_equal(s, so)

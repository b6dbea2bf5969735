"""The coded double kernels (groups of four 9-node blocks, lines by parity
class): block counts of every remainder modulo four, every level count, ROI
tiers per block of a group, and fields so large that sums of four values, or of
eight, overflow."""
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


def _huge_field(kind, shape):
    p = 2.0 ** 1022
    u = np.full(shape, 0.6 * p)  # a sum of four is finite, one of eight is not
    if kind == "peak":  # the largest value above 2^1022, alone
        u[:] = 0.9 * p
        u[3, 5, 7] = 1.05 * p
    return u


@pytest.mark.parametrize("B,K", [(9, 1), (9, 3), (17, 1), (17, 4)])
@pytest.mark.parametrize("kind", ["flat", "peak"])
def test_fields_whose_sums_of_eight_overflow(kind, B, K):
    """The oracle codes these fields, and so must the kernels, in both
    directions (check_stream_parity decodes and checks the bound)."""
    import paper_2609_00205_gb300 as bm

    # whole blocks for several levels: the zeros around a field make its coarse
    # values overshoot, and a sum of four of them must stay finite
    u = _huge_field(kind, (20, 19, 21) if K == 1 else (2 * B, B, 3 * B))
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-3, block=B, levels=K, global_levels=1).cpu().numpy()
    assert not oracle.stream_header(s)["raw"]
    check_stream_parity(bm, u, s, 1e-3, "rel", B, K, 1, label=f"f64_huge_{kind}_{B}_{K}")

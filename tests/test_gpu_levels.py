"""The global levels' passes at the edges of their dispatch: the first pass with
the coefficients taken in it (lines enough to fill the SMs, tiles of 8 or 4
lines and of 32 or 16) and apart from it, odd and even line extents around a
warp's width, dimensions of two nodes, which only copy; against the oracle."""
import numpy as np
import pytest
import torch

import fields
import oracle
from _util import check_stream_parity

pytestmark = pytest.mark.gpu

# (shape, block, levels): the first global grid has 9 nodes of 17, 5 of 9
CASES = [((136, 119, 41), 17, 1), ((119, 136, 60), 17, 1), ((68, 51, 120), 17, 1), ((400, 170, 3), 9, 1),
         ((2, 70, 1200), 17, 1), ((170, 2, 600), 17, 1)]


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("shape,B,K", CASES)
def test_streams_and_fields(shape, B, K, dt):
    import paper_2609_00205_gb300 as bm

    u = np.random.default_rng(sum(shape)).normal(size=shape).cumsum(axis=-1).astype(dt)
    t = torch.from_numpy(u).to("cuda")
    s = bm.compress(t, 1e-3, block=B, levels=K, global_levels=3).cpu().numpy()
    check_stream_parity(bm, u, s, 1e-3, "rel", B, K, 3, label=f"levels_{shape}")
    c = bm.decompose(t, block=B, levels=K, global_levels=3)
    want = oracle.decompose(u.astype(np.float64), B, K, 3)
    eps = np.finfo(dt).eps
    # a few dozen roundings of values of the field's size in each of the levels
    bound = 64 * eps * np.abs(u).max()
    assert np.abs(c.cpu().numpy() - want).max() <= bound
    assert (bm.recompose(c, shape, B, K, 3).cpu() - torch.from_numpy(u)).abs().max().item() <= bound


@pytest.mark.parametrize("shape", [(198, 200, 66), (198, 190, 70)])
def test_coefficients_by_rows_and_by_nodes(shape):
    """Whole-grid in-cache levels (8-node blocks) of 200 x 200 rows, where a warp
    takes a row's coefficients, and of 200 x 192, where a thread takes a node's."""
    import paper_2609_00205_gb300 as bm

    u = fields.power_law_grf(shape, exponent=-3.0, seed=8, dtype=torch.float64).float().numpy()
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-3, block=8, levels=2, global_levels=1).cpu().numpy()
    check_stream_parity(bm, u, s, 1e-3, "rel", 8, 2, 1, label=f"rows_{shape}")

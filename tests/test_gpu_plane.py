"""The fused 2-D block kernels: every block size and level count they take, the
two axes in any position of a 3-D shape, ragged edges around a CTA's group of
blocks (7 of 17 nodes, 14 of 9), ROI tiers and wide codes, against the oracle;
and against the whole-grid passes, which the full-precision entry points keep:
the codes are those of the coefficients that bm_decompose returns."""
import numpy as np
import pytest
import torch

import fields
from _util import check_stream_parity

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2), (9, 300), (300, 9), (17, 119), (18, 120), (65, 64), (1, 40, 77), (40, 1, 77), (40, 77, 1)]


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("B,K", [(9, 1), (9, 2), (9, 3), (17, 1), (17, 2), (17, 3), (17, 4)])
def test_planes_against_the_oracle(B, K, dt):
    import paper_2609_00205_gb300 as bm

    for i, shape in enumerate(SHAPES):
        u = np.random.default_rng(i).normal(size=shape).cumsum(axis=-1).astype(dt)
        for tol in (1e-2, 1e-5):
            s = bm.compress(torch.from_numpy(u).to("cuda"), tol, block=B, levels=K, global_levels=1).cpu().numpy()
            check_stream_parity(bm, u, s, tol, "rel", B, K, 1, label=f"plane_{shape}_{B}_{K}")


@pytest.mark.parametrize("B", [9, 17])
def test_roi_tiers_of_a_plane(B):
    import paper_2609_00205_gb300 as bm

    shape = (83, 131)
    u = fields.power_law_grf(shape, exponent=-2.5, seed=B, dtype=torch.float32).numpy()
    nb = int(np.prod([-(-n // B) for n in shape]))
    roi = np.array([1e-3, 1e-5, 1e-2])[np.arange(nb) * 5 % 3]
    s = bm.compress(torch.from_numpy(u).to("cuda"), 1e-2, roi=roi, block=B, levels=2, global_levels=2).cpu().numpy()
    check_stream_parity(bm, u, s, 1e-2, "rel", B, 2, 2, roi=roi, label=f"plane_roi_{B}")


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("B,K", [(9, 3), (17, 2)])
def test_codes_are_those_of_the_full_precision_coefficients(B, K, dt):
    """Bit for bit: the fused kernel's codes against the quantiser applied to
    the whole-grid passes' coefficients."""
    import oracle
    import paper_2609_00205_gb300 as bm

    u = np.random.default_rng(7).normal(size=(211, 187)).cumsum(axis=0).astype(dt)
    t = torch.from_numpy(u).to("cuda")
    s = bm.compress(t, 1e-3, block=B, levels=K, global_levels=0)
    h = oracle.stream_header(s.cpu().numpy())
    assert not h["raw"]
    codes = bm.stream_codes(s).cpu().numpy()
    q = s.cpu().numpy()[h["off_qtab"]:][: 8 * (K + 1)].view("<f8")
    coef = bm.decompose(t, block=B, levels=K, global_levels=0).cpu().numpy()
    n, per, cnt = B, [], []
    for _ in range(K):
        c = (n + 1) // 2
        cnt.append(n * n - c * c)
        n = c
    nblk = int(np.prod([-(-m // B) for m in u.shape]))
    width = np.concatenate([np.tile(np.concatenate([np.full(c, q[l]) for l, c in enumerate(cnt)]), nblk),
                            np.full(coef.size - nblk * sum(cnt), q[K])])
    ref, _ = oracle.quantize_array(coef.astype(np.float64), width, dt == np.float64)
    np.testing.assert_array_equal(codes, ref)

"""A batch of shapes the process has not met before: the level tables of every
new shape are uploaded inside the call, and the kernels of its items run on
streams that do not wait for the default stream.  The first call's streams
must be those of single calls."""
import pytest
import torch

import fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_first_batch_of_new_shapes(seed):
    import paper_2609_00205_gb300 as bm

    shapes = [(131 + 17 * seed + 3 * i, 207 + 29 * seed + 5 * i) for i in range(16)]
    us = [fields.power_law_grf(s, seed=40 + i, dtype=torch.float32, device="cuda").contiguous()
          for i, s in enumerate(shapes)]
    torch.cuda.synchronize()
    first = bm.compress_batch(us, [1e-3] * len(us))
    for u, s in zip(us, first):
        assert torch.equal(bm.compress(u, 1e-3), s)

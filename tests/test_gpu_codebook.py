"""The Huffman codebook above 8192 present symbols (sorted and emitted on many
CTAs, its tree built in shared-memory tiles of 20,480 merged ranks), through
the compressor: fields whose codes are drawn to given counts, at the edges of
the tiles, of the segments and of the symbols kept in shared memory.  Streams
must decode to the field within the bound and carry the oracle's lengths."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _counts(kind, n, rng):
    if kind == "equal":
        return np.full(n, 7)
    if kind == "ramp":
        return 1 + np.arange(n) % 1000
    if kind == "skewed":  # a few heavy symbols over a long tail of singletons
        c = np.ones(n, dtype=np.int64)
        c[rng.choice(n, 64, replace=False)] = 2 ** rng.integers(8, 20, 64)
        return c
    return rng.integers(1, 3, n)  # ties between leaves and pairs


@pytest.mark.parametrize("kind", ["equal", "ramp", "skewed", "ties"])
@pytest.mark.parametrize("n", [8193, 10240, 20480, 20482, 40961, 65535, 65536])
def test_lengths_above_the_shared_memory_limit(n, kind):
    import paper_2609_00205_gb300 as bm

    rng = np.random.default_rng(n)
    present = np.sort(rng.choice(65536, n, replace=False))
    sym = np.repeat(present, _counts(kind, n, rng)).astype(np.uint16)
    rng.shuffle(sym)
    so, mo = oracle.huffman_encode(sym, 65536, 2048)
    sg, mg = bm.huffman_encode(torch.from_numpy(sym.view(np.int16)).to("cuda"), 65536, 2048)
    assert mg == mo
    np.testing.assert_array_equal(sg.cpu().numpy(), so)


@pytest.mark.parametrize("scale", [2000.0, 6000.0, 30000.0])
def test_many_cta_codebook_of_a_compress_call(scale):
    """White noise quantised so that about 17,000, 45,000 and all 65,000 symbols
    are present: the cooperative sort and emission of a single call."""
    import paper_2609_00205_gb300 as bm

    g = torch.Generator().manual_seed(3)
    u = torch.randn(90, 91, 92, generator=g, dtype=torch.float32).numpy()
    tol = float(np.abs(u).max()) / scale
    so = oracle.compress(u, tol, rel=False, B=9, K=1, M=0)
    sg = bm.compress(torch.from_numpy(u).to("cuda"), tol, mode="abs", block=9, levels=1, global_levels=0).cpu().numpy()
    ho, hg = oracle.stream_header(so), oracle.stream_header(sg)
    assert not ho["raw"] and not hg["raw"]
    codes = bm.stream_codes(torch.from_numpy(sg.copy()).to("cuda")).cpu().numpy()
    s16 = np.where(np.abs(codes) < 32768, codes + 32768, 0).astype(np.uint16)
    assert len(np.unique(s16)) > 8192
    # the codebook section is that of the oracle's Huffman stage on these codes
    sec, meta = oracle.huffman_encode(s16, 65536, 2048)
    off = 8 * ((4 * meta["n_chunks"] + 7) // 8) + 8 * ((14 * meta["n_chunks"] + 7) // 8)
    got = sg[hg["off_codebook"]:hg["off_codebook"] + meta["codebook_bytes"]]
    np.testing.assert_array_equal(got, sec[off:off + meta["codebook_bytes"]])
    d = bm.decompress(torch.from_numpy(sg.copy()).to("cuda")).cpu().numpy()
    assert np.abs(d.astype(np.float64) - u).max() <= tol


@pytest.mark.parametrize("kind", ["equal", "ramp", "skewed", "ties", "doubling"])
@pytest.mark.parametrize("n", [1, 2, 3, 31, 33, 64, 1023, 1024, 1025, 2049, 7169, 8191, 8192])
def test_lengths_in_shared_memory(n, kind):
    """The tree of one block: rows of the sort, a thread's ranks of a round, and
    rounds of a single pair (counts that double)."""
    import paper_2609_00205_gb300 as bm

    rng = np.random.default_rng(n)
    present = np.sort(rng.choice(65536, n, replace=False))
    if kind == "doubling":
        counts = 2 ** np.minimum(np.arange(n), 19)[rng.permutation(n)] if n <= 64 else 1 + (np.arange(n) % 20 == 0) * 300
        counts = np.minimum(counts, 2 ** 19)
    elif kind == "skewed" and n < 64:
        counts = 2 ** rng.integers(0, 18, n)
    else:
        counts = _counts(kind, n, rng)
    sym = np.repeat(present, counts).astype(np.uint16)
    rng.shuffle(sym)
    so, mo = oracle.huffman_encode(sym, 65536, 2048)
    sg, mg = bm.huffman_encode(torch.from_numpy(sym.view(np.int16)).to("cuda"), 65536, 2048)
    assert mg == mo
    np.testing.assert_array_equal(sg.cpu().numpy(), so)

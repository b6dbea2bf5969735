"""The Huffman decoder at its edges: codebook sections of many short runs (in
several batches, and too long for the shared-memory copy), long runs, both
launch shapes (few and many runs of symbols), prefixes with codes of several
lengths, and codebook sections damaged on the host."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _round_trip(sym, dict_size, chunk):
    import paper_2609_00205_gb300 as bm

    so, mo = oracle.huffman_encode(sym, dict_size, chunk)
    back = bm.huffman_decode(torch.from_numpy(so.copy()).to("cuda"), mo, sym.size, dict_size, chunk)
    np.testing.assert_array_equal(back.cpu().numpy().view(np.uint16), sym)
    return so, mo


@pytest.mark.parametrize("stride,offset", [(2, 0), (3, 1), (7, 5), (64, 63)])
def test_codebooks_of_short_runs(stride, offset):
    """Every stride-th symbol of the dictionary: one run per symbol (32,768
    runs, a 393 KB section, at stride 2)."""
    rng = np.random.default_rng(stride)
    present = np.arange(offset, 65536, stride)
    sym = np.concatenate([present, rng.choice(present, 60_000)]).astype(np.uint16)
    rng.shuffle(sym)
    _round_trip(sym, 65536, 2048)


@pytest.mark.parametrize("n_present", [1, 2, 1023, 1024, 1025, 8192, 8193, 65536])
def test_one_run(n_present):
    rng = np.random.default_rng(n_present)
    sym = np.concatenate([np.arange(n_present), rng.integers(0, n_present, 5000)]).astype(np.uint16)
    _round_trip(sym, 65536, 1024)


@pytest.mark.parametrize("first,last", [(0, 0), (1, 40), (30_000, 30_700), (65_535, 65_535), (40_000, 65_535)])
@pytest.mark.parametrize("step", [1, 3])
def test_codebooks_anywhere_in_the_dictionary(first, last, step):
    """The canonical order is counted between the first and the last present
    symbol only."""
    present = np.unique(np.append(np.arange(first, last + 1, step), last))
    rng = np.random.default_rng(first)
    p = 0.7 ** np.minimum(np.arange(present.size), 60)
    sym = np.concatenate([present, rng.choice(present, 5000, p=p / p.sum())]).astype(np.uint16)
    _round_trip(sym, 65536, 2048)


@pytest.mark.parametrize("chunk,chunks", [(64, 14_591), (64, 14_592), (256, 15_001)])
def test_launch_shapes(chunk, chunks):
    """Around the chunk count from which one large CTA per SM decodes (three
    quarters of 152 x 1024 runs), with geometric counts: codes of 1 to about 20
    bits, so prefixes of several lengths."""
    rng = np.random.default_rng(chunks)
    sym = np.minimum(rng.geometric(0.5, chunk * chunks - 11) - 1, 255).astype(np.uint16)
    _round_trip(sym, 256, chunk)


def test_damaged_codebooks_are_refused_or_decoded():
    import paper_2609_00205_gb300 as bm

    rng = np.random.default_rng(9)
    sym = np.minimum(rng.geometric(0.05, 20_000) * 3, 4095).astype(np.uint16)
    so, mo = oracle.huffman_encode(sym, 4096, 2048)
    cb = 8 * ((4 * mo["n_chunks"] + 7) // 8) + 8 * ((14 * mo["n_chunks"] + 7) // 8)  # after chunk words and splits
    first = so.copy()
    first[cb:cb + 4] = 255  # a run beyond the dictionary
    with pytest.raises(bm.BlockMGARDError) as e:
        bm.huffman_decode(torch.from_numpy(first).to("cuda"), mo, sym.size, 4096, 2048)
    assert e.value.status == 4
    for _ in range(20):
        bad = so.copy()
        bad[cb + int(rng.integers(0, mo["codebook_bytes"]))] ^= 1 << int(rng.integers(0, 8))
        try:
            bm.huffman_decode(torch.from_numpy(bad).to("cuda"), mo, sym.size, 4096, 2048)
        except bm.BlockMGARDError as err:
            assert err.status == 4
    torch.cuda.synchronize()
    _round_trip(sym, 4096, 2048)


def _present(kind, n_runs, rng):
    """Symbols of n_runs runs: of one symbol, of a few, or with long ones among
    them (255 to 700 symbols, around the limit of a thread's own copy)."""
    if kind == "ones":
        return np.arange(n_runs) * 2
    lens = rng.integers(1, 5, n_runs)
    if kind == "long":
        at = rng.choice(n_runs, 24, replace=False)
        lens[at] = rng.integers(255, 700, 24)
        lens[at[:3]] = (255, 256, 257)
    gaps = 1 + rng.integers(0, 3, n_runs)
    first = np.cumsum(np.concatenate([[0], lens[:-1] + gaps[:-1]]))
    return np.concatenate([np.arange(f, f + c) for f, c in zip(first, lens) if f + c <= 65536])


@pytest.mark.parametrize("kind", ["ones", "few", "long"])
@pytest.mark.parametrize("n_runs", [512, 513, 514, 1000, 2731, 8000, 10922, 10923])
def test_run_headers_side_by_side(kind, n_runs):
    """Around the run count from which the headers are walked in segments, and
    the section size (10,922 runs of one symbol) up to which they are."""
    rng = np.random.default_rng(n_runs)
    present = _present(kind, n_runs, rng)
    sym = np.concatenate([present, rng.choice(present, 9000)]).astype(np.uint16)
    rng.shuffle(sym)
    _round_trip(sym, 65536, 512)


@pytest.mark.parametrize("word,value", [(0, 60000), (1, 65537), (1, 0xFFFFFFFF), (1, 40000), (3 * 777, 0), (3 * 777, 65536),
                                        (3 * 777 + 1, 4), (3 * 777 + 1, 0), (3 * 1999 + 1, 0xFFFFFFF0), (3 * 777 + 2, 33)])
def test_damaged_headers_of_many_runs(word, value):
    """One word of a section of 2,000 runs of one symbol changed on the host: an
    error, and the context stays usable.  (The symbols are three apart: a count
    of 3 takes the padding as lengths of 0 and overlaps nothing, which is a
    valid section; 4 is the least that is not.)"""
    import paper_2609_00205_gb300 as bm

    rng = np.random.default_rng(word)
    present = np.arange(2000) * 3 + 100
    sym = np.concatenate([present, rng.choice(present, 9000)]).astype(np.uint16)
    so, mo = oracle.huffman_encode(sym, 65536, 512)
    assert mo["n_runs"] == 2000 and mo["codebook_bytes"] == 24000
    off = (4 * mo["n_chunks"] + 7) // 8 * 8 + (14 * mo["n_chunks"] + 7) // 8 * 8
    bad = so.copy()
    bad[off:off + 24000].view(np.uint32)[word] = value
    with pytest.raises(bm.BlockMGARDError) as e:
        bm.huffman_decode(torch.from_numpy(bad).to("cuda"), mo, sym.size, 65536, 512)
    assert e.value.status == 4
    back = bm.huffman_decode(torch.from_numpy(so).to("cuda"), mo, sym.size, 65536, 512)
    np.testing.assert_array_equal(back.cpu().numpy().view(np.uint16), sym)


@pytest.mark.parametrize("n_runs,step", [(40, 1400), (600, 100), (11_000, 5)])
@pytest.mark.parametrize("what", ["first", "count", "order", "length", "long length"])
def test_damaged_sections_walked_in_batches(n_runs, step, what):
    """Few runs, and a section too long for the shared-memory copy (several
    batches of headers): every check of a batch refuses the stream."""
    import paper_2609_00205_gb300 as bm

    lens = np.ones(n_runs, np.int64)
    if what == "long length":
        lens[1] = 1200  # a run that the whole block copies
    first = np.concatenate([[0], np.cumsum(np.maximum(lens, step - 3)[:-1] + 3)])
    keep = first + lens <= 65536
    n_runs, first, lens = int(keep.sum()), first[keep], lens[keep]
    present = np.concatenate([np.arange(f, f + c) for f, c in zip(first, lens)])
    rng = np.random.default_rng(n_runs)
    sym = np.concatenate([present, rng.choice(present, 9000)]).astype(np.uint16)
    so, mo = oracle.huffman_encode(sym, 65536, 512)
    assert mo["n_runs"] == n_runs and (n_runs <= 600 or mo["codebook_bytes"] > 128 * 1024)
    cb = (4 * mo["n_chunks"] + 7) // 8 * 8 + (14 * mo["n_chunks"] + 7) // 8 * 8
    run = 1 if what == "long length" else n_runs - 2
    at = cb + int((8 + (lens[:run] + 3) // 4 * 4).sum())
    bad = so.copy()
    h = bad[at:at + 8].view(np.uint32)
    if what == "first":
        h[0] = 65536
    elif what == "count":
        h[1] = 65537
    elif what == "order":
        h[0] = first[run - 1]
    else:
        bad[at + 8 + int(lens[run]) - 1] = 33
    with pytest.raises(bm.BlockMGARDError) as e:
        bm.huffman_decode(torch.from_numpy(bad).to("cuda"), mo, sym.size, 65536, 512)
    assert e.value.status == 4
    back = bm.huffman_decode(torch.from_numpy(so).to("cuda"), mo, sym.size, 65536, 512)
    np.testing.assert_array_equal(back.cpu().numpy().view(np.uint16), sym)

"""The Huffman encoder at the edges of its tiles: chunk sizes of whole and
partial 256-symbol steps, symbol counts around a tile of chunks, each of its
tables (small window, split table of the whole dictionary, codes too long for
a window entry); every section must be the oracle's byte for byte."""
import numpy as np
import pytest
import torch

import fields
import oracle

pytestmark = pytest.mark.gpu


def _check(sym, dict_size, chunk):
    import paper_2609_00205_gb300 as bm

    so, mo = oracle.huffman_encode(sym, dict_size, chunk)
    sg, mg = bm.huffman_encode(torch.from_numpy(sym.view(np.int16)).to("cuda"), dict_size, chunk)
    assert mg == mo
    np.testing.assert_array_equal(sg.cpu().numpy(), so)
    back = bm.huffman_decode(sg, mg, sym.size, dict_size, chunk)
    np.testing.assert_array_equal(back.cpu().numpy().view(np.uint16), sym)


@pytest.mark.parametrize("dict_size", [8192, 65536])
@pytest.mark.parametrize("chunk", [64, 96, 256, 512, 768, 1280, 1792, 2016, 2048])
def test_chunk_sizes(chunk, dict_size):
    sym = fields.laplace_symbols(9 * chunk + 37, dict_size // 2, dict_size / 20, seed=chunk, escape_rate=0.01)
    _check(sym, dict_size, chunk)


@pytest.mark.parametrize("dict_size,scale", [(4096, 1.0), (65536, 9000.0)])
@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 4 * 2048 - 1, 4 * 2048, 8 * 2048, 8 * 2048 + 1,
                               3 * 8 * 2048 + 5])
def test_symbol_counts_around_tiles(n, dict_size, scale):
    _check(fields.laplace_symbols(n, dict_size // 2, scale, seed=n), dict_size, 2048)


@pytest.mark.parametrize("dict_size,scale", [(4096, 1.0), (4096, 300.0), (65536, 9000.0)])
@pytest.mark.parametrize("chunk,over", [(64, 0), (64, 1), (512, 1)])
def test_short_and_long_streams(chunk, over, dict_size, scale):
    """At and above the chunk count (eight per SM of 152) up to which one
    launch codes with the table left in global memory."""
    n = 8 * 152 * chunk + over
    _check(fields.laplace_symbols(n, dict_size // 2, scale, seed=n), dict_size, chunk)


def test_short_stream_of_long_codes():
    """29 symbols with Fibonacci counts: codes of up to 28 bits."""
    f = [1, 1]
    while len(f) < 29:
        f.append(f[-1] + f[-2])
    sym = np.repeat(np.arange(3, 3 + len(f)), f).astype(np.uint16)
    np.random.default_rng(6).shuffle(sym)
    _check(sym, 4096, 2048)


@pytest.mark.parametrize("dict_size", [128, 16384])
def test_codes_longer_than_a_window_entry(dict_size):
    """Fibonacci counts (36 symbols, 39 M in all) give codes of 1 to 35 bits,
    limited to 32: longer than the 27 bits of a window entry in a dictionary
    that fits the small window."""
    f = [1, 1]
    while len(f) < 36:
        f.append(f[-1] + f[-2])
    rng = np.random.default_rng(5)
    sym = np.repeat(np.arange(3, 3 + len(f)), f).astype(np.uint16)
    rng.shuffle(sym)
    _check(sym, dict_size, 2048)


def test_short_stream_with_codes_too_long_for_an_entry():
    """A stream short enough for the encoder without a table of its own, whose
    codes are up to 28 bits: 29 values with Fibonacci counts."""
    import paper_2609_00205_gb300 as bm

    shape, B, K, M = (119, 119, 119), 17, 2, 1
    n = bm.coeff_count(shape, B, K, M)
    fib = [1, 1]
    while len(fib) < 29:
        fib.append(fib[-1] + fib[-2])
    values = np.repeat(np.arange(29) - 14, fib)
    codes = np.full(n, 14, np.int64)  # the most frequent
    codes[: values.size] = values
    codes = np.random.default_rng(0).permutation(codes)
    # the bin widths of the levels, from a stream of the same shape and tolerance
    probe = bm.compress(torch.from_numpy(np.random.default_rng(1).normal(size=shape)).to("cuda"), 1.0, mode="abs",
                        block=B, levels=K, global_levels=M).cpu().numpy()
    h = oracle.stream_header(probe)
    q = probe[h["off_qtab"]:][: 8 * (K + M + 1)].view("<f8")
    per = [B ** 3 - 9 ** 3, 9 ** 3 - 5 ** 3]
    nb = 7 ** 3
    width = np.tile(np.repeat(q[:K], per), nb)
    gcount = 35 ** 3 - 18 ** 3
    width = np.concatenate([width, np.full(gcount, q[K]), np.full(n - width.size - gcount, q[K + 1])])
    u = bm.recompose(torch.from_numpy(codes * width).to("cuda"), shape, B, K, M)
    s = bm.compress(u, 1.0, mode="abs", block=B, levels=K, global_levels=M)
    got = bm.stream_codes(s).cpu().numpy()
    np.testing.assert_array_equal(got, codes)  # the bins are far wider than the roundings
    hs = oracle.stream_header(s.cpu().numpy())
    so, mo = oracle.huffman_encode((codes + 32768).astype(np.uint16), 65536, 2048)
    assert mo["n_words"] == hs["n_words"] and mo["n_runs"] == hs["n_runs"]
    words = s.cpu().numpy()[hs["off_bits"]:][: 4 * hs["n_words"]]
    off = sum(-(-b // 8) * 8 for b in (4 * mo["n_chunks"], 14 * mo["n_chunks"], mo["codebook_bytes"]))
    np.testing.assert_array_equal(words, so[off:][: 4 * mo["n_words"]])


@pytest.mark.parametrize("dict_size", [8192, 8194, 65536])
@pytest.mark.parametrize("off", [1, 3, 7])
def test_symbols_at_any_address(off, dict_size):
    """Symbols that start between 16-byte boundaries, fewer and more of them
    than reach the first boundary."""
    import paper_2609_00205_gb300 as bm

    rng = np.random.default_rng(off)
    for n in (1, 8 - off, 9, 5003, 8 * 2048):
        sym = rng.integers(0, dict_size, n).astype(np.uint16)
        so, mo = oracle.huffman_encode(sym, dict_size, 2048)
        buf = torch.empty(n + 8, dtype=torch.int16, device="cuda")
        d = buf[off:off + n]
        d.copy_(torch.from_numpy(sym.view(np.int16)))
        sg, mg = bm.huffman_encode(d, dict_size, 2048)
        assert mg == mo
        np.testing.assert_array_equal(sg.cpu().numpy(), so)

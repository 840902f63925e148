"""The Huffman decoder's branches at the sizes where they change: tables held
in shared memory or read from global (a CTA's subsequences span more than two
images), entries that hold values or rows of the stored table (and images of
both kinds side by side), 8 or 9 warps a CTA, codewords of one bit (256 symbols
a subsequence) and of twelve, precisions below a vector load's width.  The
symbols that were coded come back exactly."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from test_huffman_gpu import _built, _gpu, _pack_batch  # noqa: F401  (_built: the module's fixture)

pytestmark = pytest.mark.gpu


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _tiny(n, p):  # n images of one subsequence or none
    r = _rng(n)
    return [np.clip(np.rint(r.laplace(0, 1.5, int(r.integers(1, 40)))), -7, 7).astype(np.int32)
            for _ in range(n)], p


def _mixed():  # small values, wide values, small values; 2,500 symbols in the middle table
    r = _rng(2)
    wide = r.permutation(np.r_[np.arange(2500) * 77777 - 90000000, r.integers(0, 9, 20000)])
    return [np.rint(r.laplace(0, 5, 9000)).astype(np.int32), wide.astype(np.int32),
            np.array([2047, -2048, 0, 0, 0] * 700, np.int32), np.array([2048, 1] * 900, np.int32)], 12


def _low_entropy():
    r = _rng(3)
    return [(r.random(300000) < 0.01).astype(np.int32), np.full(50000, 9, np.int32)], 12


def _unsynchronising():  # 12-bit codewords, 256-bit subsequences: decodings from a wrong bit stay wrong
    return [_rng(3).integers(0, 4096, 30000).astype(np.int32) - 2048], 12


def _short(p):  # every length is p, or nearly
    r = _rng(p)
    return [r.integers(0, 2 ** p, s).astype(np.int32) for s in (1, 255, 4000)], p


CASES = {"tiny200": lambda: _tiny(200, 6), "tiny2000": lambda: _tiny(2000, 4), "mixed": _mixed,
         "low_entropy": _low_entropy, "p1": lambda: _short(1), "p2": lambda: _short(2),
         "p8": lambda: _short(8)}


@pytest.mark.parametrize("name", CASES)
def test_ranges(name):
    syms, p = CASES[name]()
    d = _pack_batch([wk.huffman_pack(s, p) for s in syms], p)
    sym_off = np.r_[0, np.cumsum([s.size for s in syms])].astype(np.int64)
    assert np.array_equal(_gpu(d, sym_off), np.concatenate(syms))


def test_a_stream_that_does_not_synchronise_is_reported():
    from paper_2609_09020_gb300 import pic
    (s,), p = _unsynchronising()
    with pytest.raises(pic.PicError):
        _gpu(_pack_batch([wk.huffman_pack(s, p)], p), np.array([0, s.size], np.int64))


@pytest.mark.parametrize("n", [22, 24, 47])
def test_rounds_of_groups(n):
    """The first n images of the 64-image batch: 8 warps a CTA and one round
    of groups, 9 warps, and two rounds."""
    h = wk.huffman_streams("c5")
    w, s = int(h["word_off"][n]), int(h["sym_off"][n])
    d = dict(words=h["words"][:w], word_off=h["word_off"][:n + 1], n_bits=h["n_bits"][:n],
             tab_value=h["tab_value"][:n], tab_len=h["tab_len"][:n], p=h["p"])
    assert np.array_equal(_gpu(d, h["sym_off"][:n + 1]), h["symbols"][:s])

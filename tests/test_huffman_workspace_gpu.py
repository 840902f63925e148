"""The two workspace sizes that the Huffman decoder takes: what
pic_huffman_workspace_bytes says, and 36 bytes a subsequence plus 2 a table
entry, which is less for batches of small images.  Buffers of exactly the
smaller size (no byte behind it is touched) and one byte below it, which is
refused; tables in shared memory and, with more images than CTAs, in global
memory, and tables whose values take more than 12 bits beside others."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from test_huffman_gpu import _built, _pack_batch  # noqa: F401  (_built: the module's fixture)

pytestmark = pytest.mark.gpu
GUARD = 4096


def small_size(n_words, B, p):
    n_sub = n_words // wk.HUFF_WORDS_PER_SUBSEQ
    head = (16 + 4 * 64 + 8 * 8192 + 2 * (B << p) + 15) // 16 * 16
    return (head + 36 * n_sub + 15) // 16 * 16


def _images(n, wide_every=0):
    r = np.random.Generator(np.random.PCG64(n))
    out = []
    for i in range(n):
        s = np.rint(r.laplace(0, 4.0, int(r.integers(1, 900)))).astype(np.int32)
        out.append(s * 100003 if wide_every and i % wide_every == 0 else s)
    return out


@pytest.mark.parametrize("n,wide_every", [(1, 0), (200, 7), (2000, 0), (700, 3)])
def test_smaller_workspace(n, wide_every):
    import torch
    from paper_2609_09020_gb300 import pic
    p, syms = 12, _images(n, wide_every)
    if n == 1:  # one 12-bit table and one subsequence
        syms = [np.arange(20, dtype=np.int32)]
    d = _pack_batch([wk.huffman_pack(s, p) for s in syms], p)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    sym_off = t(np.r_[0, np.cumsum([s.size for s in syms])].astype(np.int64))
    words, word_off, n_bits = t(d["words"].view(np.int32)), t(d["word_off"]), t(d["n_bits"])
    tv, tl = t(d["tab_value"]), t(d["tab_len"])
    want = np.concatenate(syms)
    size = small_size(words.numel(), n, p)
    full = pic.pic_huffman_workspace_bytes(words.numel(), n, p)
    assert (size < full) == (n > 1)
    s = torch.cuda.current_stream().cuda_stream

    def decode(nbytes):
        ws = torch.full((max(size, full) + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
        out = torch.full((want.size,), 77, dtype=torch.int32, device="cuda")
        rc = pic.pic_huffman_decode(words.data_ptr(), words.numel(), word_off.data_ptr(), n_bits.data_ptr(), n,
                                    tv.data_ptr(), tl.data_ptr(), tv.shape[1], p, sym_off.data_ptr(), out.data_ptr(),
                                    ws.data_ptr(), nbytes, s)
        if rc == pic.PIC_OK:
            assert pic.pic_huffman_status(ws.data_ptr(), s) == pic.PIC_OK
            assert bool((ws[nbytes:] == 0xA5).all())
        return rc, out.cpu().numpy()

    for nbytes in {size, full}:
        rc, got = decode(nbytes)
        assert rc == pic.PIC_OK and np.array_equal(got, want), nbytes
    rc, got = decode(min(size, full) - 1)
    assert rc == pic.PIC_ERR_INVALID_ARG and (got == 77).all()

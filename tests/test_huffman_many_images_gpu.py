"""Huffman batches of more images than the decoder has CTAs, whose tables a
launch of their own makes: image counts on both sides of that line, tiny images
(for which no table of windows is made) and larger ones, narrow and wide values,
and the report of a bad table, which the next call on the same workspace does
not keep."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from test_huffman_gpu import _built, _pack_batch  # noqa: F401  (_built: the module's fixture)

pytestmark = pytest.mark.gpu


def _images(n, most, p):
    r = np.random.Generator(np.random.PCG64(n + most))
    top = 2 ** (p - 1) // 3 + 1
    out = [np.clip(np.rint(r.laplace(0, 3.0, int(r.integers(1, most + 1)))), -top, top).astype(np.int32) for _ in range(n)]
    out[n // 2] = out[n // 2] * 70001  # one image of wide values
    return out


@pytest.mark.parametrize("most", [25, 900])
@pytest.mark.parametrize("n,p", [(600, 12), (620, 12), (2000, 12), (620, 1), (620, 5), (3000, 8)])
def test_many_images(n, p, most):
    import torch
    from paper_2609_09020_gb300 import pic
    syms = [np.full(min(most, 40), 6, np.int32)] * n if p == 1 else _images(n, most, p)
    d = _pack_batch([wk.huffman_pack(s, p) for s in syms], p)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    sym_off = t(np.r_[0, np.cumsum([s.size for s in syms])].astype(np.int64))
    words, word_off, n_bits = t(d["words"].view(np.int32)), t(d["word_off"]), t(d["n_bits"])
    tv = t(d["tab_value"])
    good, bad = t(d["tab_len"]), d["tab_len"].copy()
    bad[n - 3, 0] = 13  # past every precision
    bad = t(bad)
    want = np.concatenate(syms)
    ws = torch.full((pic.pic_huffman_workspace_bytes(words.numel(), n, p),), 0xA5, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for tl, status in ((good, pic.PIC_OK), (bad, pic.PIC_ERR_INVALID_ARG), (good, pic.PIC_OK)):
        out = torch.full((want.size,), 77, dtype=torch.int32, device="cuda")
        assert pic.pic_huffman_decode(words.data_ptr(), words.numel(), word_off.data_ptr(), n_bits.data_ptr(), n,
                                      tv.data_ptr(), tl.data_ptr(), tv.shape[1], p, sym_off.data_ptr(), out.data_ptr(),
                                      ws.data_ptr(), ws.numel(), s) == pic.PIC_OK
        assert pic.pic_huffman_status(ws.data_ptr(), s) == status
        if status == pic.PIC_OK:
            assert np.array_equal(out.cpu().numpy(), want)

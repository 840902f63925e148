"""Inverse ZpR on streams whose blocks differ in length along the stream: a
2,048-symbol chunk of empty blocks writes fifty times what one of long blocks
does, so neighbouring chunks must not fall to one CTA.  Values and offsets
against the blocks that were coded, on streams of one chunk to several per CTA
and at any alignment; and the time of a stream whose flat blocks lie together
against one with the same blocks mixed (1.1 times where chunks are dealt out in
turn, 2.8 where each CTA takes a contiguous range: the bound is 1.8)."""
import pytest

pytestmark = pytest.mark.gpu
EOB = 272


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build
    build.build()


def _stream(parts, skip=0):
    """(blocks, literals each) parts -> symbols (`skip` words into their buffer), coefficients, offsets."""
    import torch
    from paper_2609_09020_gb300 import pic  # noqa: F401
    from perf.cases import _zz_order
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    order = torch.tensor(_zz_order(), device="cuda")
    syms, coeffs = [], []
    for n, lits in parts:
        s = torch.randint(1, 200, (n, lits + 1), generator=g, device="cuda", dtype=torch.int32)
        s[:, lits] = EOB
        zz = torch.zeros((n, 64), dtype=torch.int32, device="cuda")
        zz[:, order[:lits]] = s[:, :lits]
        syms.append(s.reshape(-1))
        coeffs.append(zz)
    syms = torch.cat(syms)
    buf = torch.zeros(syms.numel() + skip, dtype=torch.int32, device="cuda")
    buf[skip:] = syms
    return buf[skip:], torch.cat(coeffs), torch.nonzero(syms == EOB)[:, 0]


def _decoder(sym, n_blocks):
    import torch
    from paper_2609_09020_gb300 import pic
    coeffs = torch.full((n_blocks, 64), 77, dtype=torch.int32, device="cuda")
    offsets = torch.full((n_blocks,), -1, dtype=torch.int64, device="cuda")
    ws = torch.empty(pic.pic_izpr_workspace_bytes(sym.numel()), dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def decode():
        assert pic.pic_izpr_decode(sym.data_ptr(), sym.numel(), EOB, n_blocks, coeffs.data_ptr(), offsets.data_ptr(),
                                   ws.data_ptr(), ws.numel(), s) == pic.PIC_OK
    return decode, coeffs, offsets, lambda: pic.pic_izpr_status(ws.data_ptr(), s)


N = 8192
STREAMS = {
    "one_chunk": [(40, 3), (500, 0), (20, 40)],
    "nine_chunks": [(200, 60), (4000, 0), (30, 64)],
    "flat_first": [(30 * N, 0), (30 * N, 30)],
    "flat_last": [(10 * N, 62), (70 * N, 0)],
    "several_chunks_a_cta": [(20 * N, 63), (9 * N, 0), (40 * N, 1), (3 * N, 64), (1, 0)],
}


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("name", STREAMS)
def test_values(name, skip):
    import torch
    from paper_2609_09020_gb300 import pic
    sym, want, marks = _stream(STREAMS[name], skip)
    decode, coeffs, offsets, status = _decoder(sym, want.shape[0])
    for _ in range(2):
        decode()
    assert status() == pic.PIC_OK
    assert torch.equal(coeffs, want) and torch.equal(offsets, marks)
    for wrong in (-1, 1):  # one block fewer or more than the stream has
        decode, coeffs, offsets, status = _decoder(sym, want.shape[0] + wrong)
        decode()
        assert status() == pic.PIC_ERR_INVALID_ARG


def test_flat_stretches_are_shared():
    import torch
    n, times = 32 * N, []
    for parts in ([(n, 0), (n, 49)], [(64, 0), (64, 49)] * (n // 64)):
        sym, want, _ = _stream(parts)
        decode, *_ = _decoder(sym, want.shape[0])
        runs = []
        for i in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                decode()
            b.record()
            b.synchronize()
            runs.append(a.elapsed_time(b))
        times.append(sorted(runs)[3])
    assert times[0] < 1.8 * times[1], times

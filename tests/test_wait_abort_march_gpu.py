"""The bounded waits of the row-marching tcgen05 kernel (what staging "auto"
runs on 64-wide nets), made to run out on purpose as in test_wait_abort_gpu.py:
one decoding warp of each group of the first CTA withholds its first arrival and
the poll limit is microseconds' worth; nothing faults, traps or hangs.  Through
the handle: the output layer on the tensor pipe and in fp32, and ranges that go
on to a second image after the abort (200 images of eight tiles on 152 CTAs)."""
import pytest

from paper_2609_09020_gb300 import workloads as wk

from decode_util import max_abs_diff, oracle_full

from test_wait_abort_gpu import P, SHORT_LIMIT, _buffers, _built  # noqa: F401  (_built: the module's fixture)

pytestmark = pytest.mark.gpu
NETS = [(7, 1, (7, 64, 64, 3), "relu"), (8, 1, (8, 64, 64, 64, 3), "relu"), (8, 2, (16, 64, 64, 64, 3), "gelu")]


@pytest.mark.parametrize("H,W,B", [(48, 384, 1), (8, 8, 200)])
@pytest.mark.parametrize("net", NETS, ids=lambda n: "x".join(map(str, n[2])))
def test_withheld_arrival_times_out_and_the_handle_recovers(orc, net, H, W, B):
    import torch
    from paper_2609_09020_gb300 import pic
    L, C, dims, act = net
    wl = wk.custom(f"abort_{H}x{W}", H, W, L, C, dims, act=act, weight_dtype="fp16", batch=B, precisions=(P,))
    x = wk.make_inputs(wl)
    lat, st, w, out = _buffers(wl, x)
    dec = pic.Decoder.for_workload(wl, P, max_batch=B)
    assert "_tile" not in dec.kernel_name and "_tma" not in dec.kernel_name
    s = torch.cuda.current_stream().cuda_stream
    for _ in range(2):
        try:
            assert pic.pic_decode_test_wait_fault(1, SHORT_LIMIT) == pic.PIC_OK
            rc = pic.pic_decode_batch(dec.handle, B, lat.data_ptr(), st.data_ptr(), w.data_ptr(), H, W,
                                      out.data_ptr(), s)
            assert rc == pic.PIC_OK
            assert pic.pic_decode_check(dec.handle, s) == pic.PIC_ERR_TIMEOUT
        finally:
            pic.pic_decode_test_wait_fault(0, 0)
        assert pic.pic_decode_check(dec.handle, s) == pic.PIC_OK  # the flag was cleared
        out.fill_(float("nan"))
        dec.decode_batch(lat, st, w, H, W, out, B=B)
        dec.check()
        got = out.cpu().numpy()
        for b in {0, 1, B - 1} & set(range(B)):
            d, where = max_abs_diff(got[b], oracle_full(orc, wl, x, b, P))
            assert d <= 2e-4, (b, d, where)
    dec.close()

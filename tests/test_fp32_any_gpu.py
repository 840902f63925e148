"""The fp32 kernel for nets without one of their own: every unrolled width
class and the padding around it, nets of 1 to 6 layers, nets too large for
the tiled kernel's shared memory, and one process decoding nets of different
shared-memory sizes in turn (one kernel function serves them).  Every pixel
against the oracle, max |error| <= 1e-4 (the fp32 path's bar)."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from decode_util import TOL, gpu_decode, max_abs_diff, oracle_full

pytestmark = pytest.mark.gpu

NETS = [
    (1, 1, (1, 3)),
    (2, 3, (6, 1, 3)),
    (3, 1, (3, 8, 9, 3)),
    (5, 1, (5, 16, 17, 24, 3)),
    (4, 2, (8, 33, 40, 3)),
    (6, 1, (6, 41, 48, 56, 3)),
    (3, 2, (6, 64, 57, 3)),
    (4, 1, (4, 65, 96, 3)),
    (12, 4, (48, 97, 3)),
    (2, 1, (2, 128, 128, 3)),
    (2, 1, (2, 7, 7, 7, 7, 7, 3)),
    (2, 1, (2, 128, 128, 128, 3)),  # beyond the tiled kernel's shared memory
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build
    build.build()


@pytest.mark.parametrize("act", ["relu", "gelu"])
@pytest.mark.parametrize("net", NETS, ids=lambda n: "x".join(map(str, n[2])))
def test_widths(orc, net, act):
    from paper_2609_09020_gb300.pic import Decoder
    L, C, dims = net
    wl = wk.custom("any", 11, 150, L, C, dims, act=act, seed=4400 + sum(dims), batch=2)
    x = wk.make_inputs(wl)
    dec = Decoder.for_workload(wl, "fp32")
    assert dec.kernel_name == "fp32_generic"
    dec.close()
    got = gpu_decode(wl, x, "fp32")
    for b in range(2):
        d, where = max_abs_diff(got[b], oracle_full(orc, wl, x, b, "fp32"))
        assert d <= TOL["fp32"], (dims, act, b, d, where)


def test_two_sizes_share_a_kernel(orc):
    """A larger net's handle still launches after a smaller net's was created
    (and the allocation-free entry point after either)."""
    import torch
    from paper_2609_09020_gb300 import pic
    wls = [wk.custom("big", 5, 140, 2, 1, (2, 128, 100, 3), seed=81), wk.custom("small", 5, 140, 2, 1, (2, 100, 3), seed=82)]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    xs = [wk.make_inputs(w) for w in wls]
    decs = [pic.Decoder.for_workload(w, "fp32") for w in wls]
    for i in (0, 1, 0):
        wl, x = wls[i], xs[i]
        want = oracle_full(orc, wl, x, 0, "fp32")
        lat, st, w = t(x.latents), t(x.steps), t(x.weights_for("fp32"))
        out = torch.empty((1, 3, wl.H, wl.W), device="cuda")
        decs[i].decode_batch(lat, st, w, wl.H, wl.W, out)
        assert max_abs_diff(out.cpu().numpy()[0], want)[0] <= TOL["fp32"]
        arch = pic.make_arch(wl.L, wl.C, wl.dims, wl.act, "fp32", True, wl.H, wl.W, 1)
        out.zero_()
        rc = pic.pic_decode_batch_noalloc(arch, 1, lat.data_ptr(), st.data_ptr(), w.data_ptr(), wl.H, wl.W,
                                          out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == pic.PIC_OK
        assert max_abs_diff(out.cpu().numpy()[0], want)[0] <= TOL["fp32"]
    for d in decs:
        d.close()

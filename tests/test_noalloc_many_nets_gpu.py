"""pic_decode_batch_noalloc on more nets than there are kernels: the fp32
kernel for nets without one of their own serves any number of them, and sets
itself up once per device, not once per net.  After each net's first call, a
further call launches and does nothing else, and decodes as the handle's
entry point does (the same kernel, hence the same bits)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
H, W = 24, 70
NETS = [(L, 1, (L, w, 3)) for L in (1, 2, 3, 4, 5) for w in (9, 17, 25, 33, 41, 49, 57, 65)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build
    build.build()


def test_every_net_is_set_up_once():
    import torch
    from paper_2609_09020_gb300 import pic
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    stream = torch.cuda.current_stream().cuda_stream
    calls = []
    for L, C, dims in NETS:
        arch = pic.make_arch(L, C, dims, "relu", "fp32", True, H, W, 1)
        lat = torch.randint(-20, 20, (1, pic.pic_latent_count(H, W, L, C)), generator=g, device="cuda",
                            dtype=torch.int32)
        w = torch.randn((1, pic.pic_param_count(arch)), generator=g, device="cuda") * 0.2
        calls.append((arch, lat, torch.ones((1, L), device="cuda"), w))

    def decode(arch, lat, steps, w):
        out = torch.full((1, 3, H, W), float("nan"), device="cuda")
        rc = pic.pic_decode_batch_noalloc(arch, 1, lat.data_ptr(), steps.data_ptr(), w.data_ptr(), H, W,
                                          out.data_ptr(), stream)
        assert rc == pic.PIC_OK
        return out.cpu().numpy()

    first = [decode(*c) for c in calls]
    setups = pic.pic_decode_test_noalloc_setups()
    again = [decode(*c) for c in calls]
    assert pic.pic_decode_test_noalloc_setups() == setups
    for (L, C, dims), (arch, lat, steps, w), a, b in zip(NETS, calls, first, again):
        dec = pic.Decoder(L, C, dims, "relu", "fp32", True, H, W, 1)
        assert dec.kernel_name == "fp32_generic"
        out = torch.full((1, 3, H, W), float("nan"), device="cuda")
        dec.decode(lat, steps, w, H, W, out)
        want = out.cpu().numpy()
        dec.close()
        assert np.isfinite(want).all()
        assert np.array_equal(a, want) and np.array_equal(b, want), dims

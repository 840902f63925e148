"""The CUDA GELU over the real line, through the fp32 decoder: a net whose
hidden layer is (z, -z) and whose output passes it on, fed one value per pixel.
Bound: the polynomial's error with the fp32 evaluation order (5.2e-7, most of
it the rounding of results near 8) plus 0.17 x 2 ulp of ex2.approx, 5.6e-7; from
Z = 5.8 on the value is max(z, 0) exactly, as it is at zero."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_gelu_values():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build, pic
    build.build()
    from math import erfc, sqrt
    z = np.concatenate([np.linspace(-8, 8, 8185), [0.0, -0.0, 1e-30, 5.8, 5.8000006, 1e4, 1e30]]).astype(np.float32)
    n = z.size
    w = np.array([1, -1, 0, 0, 1, 0, 0, 1, 0, 0, 0, 0, 0], np.float32)  # (z, -z), then both as they are
    dec = pic.Decoder(1, 1, (1, 2, 3), "gelu", "fp32", False, 1, n, 1, "fp32")
    t = lambda a: torch.from_numpy(a).cuda()
    out = torch.empty(1, 3, 1, n, device="cuda")
    dec.decode_batch(t(z[None]), t(np.ones((1, 1), np.float32)), t(w[None]), 1, n, out)
    got = out.cpu().numpy()[0, :, 0].astype(np.float64)
    dec.close()
    for row, s in ((0, z), (1, -z)):
        want = np.array([max(v, 0.0) - abs(v) * 0.5 * erfc(abs(v) / sqrt(2)) for v in s.astype(np.float64)])
        near = np.abs(s) <= 8
        assert np.max(np.abs(got[row] - want)[near]) <= 5.6e-7
        far = np.abs(s) >= np.float32(5.8)
        assert np.array_equal(got[row][far], np.maximum(s, 0)[far].astype(np.float64))
        assert not got[row][s == 0].any()

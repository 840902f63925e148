"""The row-marching tensor-core kernels at the edges of what they split work
by: strips of 32 and tiles of 128 columns, tables of 32 rows, runs that start
in mid-column, feature sets and groups with an odd or no tile, several images
per CTA, both latent formats.  Every pixel against the oracle on the weights
the kernel consumes, within the split's own bound (2e-4; the path's bar is
4e-3)."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from decode_util import ORACLE_THREADS, gpu_decode, max_abs_diff, oracle_full

pytestmark = pytest.mark.gpu
P = "fp16_tc"
BOUND = 2e-4

NETS = [
    (4, 1, (4, 16, 16, 3), "relu", True),
    (7, 1, (7, 40, 40, 3), "gelu", True),
    (7, 2, (14, 64, 64, 3), "relu", True),
    (8, 2, (16, 64, 64, 64, 3), "gelu", True),
    (7, 1, (7, 64, 64, 3), "relu", True),
    (8, 1, (8, 8, 8, 8, 3), "relu", False),
    (8, 1, (8, 16, 16, 16, 3), "relu", False),
    (8, 1, (8, 32, 32, 32, 3), "relu", False),
    (8, 1, (8, 64, 64, 64, 3), "relu", False),
]
SHAPES = [(1, 1, 1), (1, 129, 1), (33, 33, 3), (65, 31, 2), (97, 130, 1), (200, 64, 5), (2, 700, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build
    build.build()


@pytest.mark.parametrize("H,W,B", SHAPES)
@pytest.mark.parametrize("net", NETS, ids=lambda n: "x".join(map(str, n[2])))
def test_edges(orc, net, H, W, B):
    L, C, dims, act, f32lat = net
    wl = wk.custom(f"march_{H}x{W}", H, W, L, C, dims, act=act, weight_dtype="fp16", seed=7100 + H + W, batch=B,
                   precisions=(P,))
    x = wk.make_inputs(wl)
    got = gpu_decode(wl, x, P)
    for b in range(B):
        d, where = max_abs_diff(got[b], oracle_full(orc, wl, x, b, P))
        assert d <= BOUND, (wl.name, b, d, where)
    if not f32lat:
        return
    import torch
    from paper_2609_09020_gb300.pic import Decoder
    rng = np.random.default_rng(H * 1000 + W)
    lat = rng.laplace(0.0, 2.0, x.latents.shape).astype(np.float32)
    dec = Decoder.for_workload(wl, P, max_batch=B, latent="fp32")
    out = torch.full((B, 3, H, W), float("nan"), device="cuda")
    dec.decode_batch(torch.from_numpy(lat).cuda(), None, torch.from_numpy(x.weights_for(P)).cuda(), H, W, out, B=B)
    dec.check()
    for b in range(B):
        want = orc.decode_values(lat[b].astype(np.float64), x.weights_for(P)[b].astype(np.float64), H, W, L, C, dims,
                                 act, nthreads=ORACLE_THREADS)
        d, where = max_abs_diff(out[b].cpu().numpy(), want)
        assert d <= BOUND, (wl.name, "fp32 latents", b, d, where)
    dec.close()

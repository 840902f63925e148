"""The output layer of narrow and of deep nets works on fp32 hidden values
(PIC_PREC_FP16_TC): fp16 operand pairs end at 131,008 and have an absolute
step of 2^-24, an fp32 value has neither limit.

The last hidden layer's weights are whole multiples of a power of two that
brings its values to 1e5 .. 1e7, or to 1e-6 .. 1e-4; the output weights bring
them back to where the pixels are.  Every pixel, unclamped, against the oracle
on the same weights, relative to the largest value.  The bound: 22 bits from
each of up to three split operands, an fp32 sum of 64 terms, and 5e-6 from the
GELU on small values, times the cancellation in the last sum (its terms'
magnitudes add up to at most 11 times the largest pixel):
11 (3 2^-21 + 64 2^-24 + 5e-6) = 1.13e-4."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from decode_util import gpu_decode, max_abs_diff, oracle_full

pytestmark = pytest.mark.gpu
P = "fp16_tc"
BOUND = 1.2e-4

NETS = [
    (4, 1, (4, 16, 16, 3), "relu"),
    (8, 1, (8, 8, 8, 8, 3), "relu"),
    (8, 1, (8, 16, 16, 16, 3), "relu"),
    (8, 1, (8, 32, 32, 32, 3), "relu"),
    (8, 1, (8, 64, 64, 64, 3), "relu"),
    (8, 2, (16, 64, 64, 64, 3), "gelu"),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_09020_gb300 import build
    build.build()


def _last_layers(w, dims, rng, hidden_exp, out_exp):
    """Replaces the last hidden layer's and the output layer's parameters (one image's, fp16)."""
    o = sum(b * (a + 1) for a, b in zip(dims[:-3], dims[1:-2]))
    for a, b, e in ((dims[-3], dims[-2], hidden_exp), (dims[-2], dims[-1], out_exp)):
        k = rng.integers(-7, 8, a * b)
        if e == hidden_exp:
            k = np.where(rng.random(a * b) < 0.7, np.abs(k), k)  # few hidden values are cut off
        w[o:o + a * b] = (k * 2.0 ** e).astype(np.float16)
        w[o + a * b:o + (a + 1) * b] = 0
        o += (a + 1) * b
    assert o == w.size and np.isfinite(w).all()


@pytest.mark.parametrize("hidden_exp,out_exp", [(13, -13), (-24, 12)], ids=["large", "small"])
@pytest.mark.parametrize("net", NETS, ids=lambda n: "x".join(map(str, n[2])))
def test_hidden_values_beyond_fp16(orc, net, hidden_exp, out_exp):
    L, C, dims, act = net
    wl = wk.custom("out_range", 37, 150, L, C, dims, act=act, weight_dtype="fp16", seed=4200, precisions=(P,))
    x = wk.make_inputs(wl)
    _last_layers(x.weights_for(P)[0], dims, np.random.default_rng(17), hidden_exp, out_exp)
    want = oracle_full(orc, wl, x, 0, P, clamp=False)
    got = gpu_decode(wl, x, P, clamp=False)[0]
    d, where = max_abs_diff(got, want)
    assert d <= BOUND * np.abs(want).max(), (d / np.abs(want).max(), where)

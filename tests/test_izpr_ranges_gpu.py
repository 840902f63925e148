"""Inverse ZpR where its ranges change: symbol counts around one chunk (2,048
symbols), around as many chunks as CTAs stay resident and a little more (ranges
of unequal length), at every alignment of the stream, and blocks that straddle
the boundaries.  The blocks that were encoded come back exactly, with the
markers' stream indexes."""
import numpy as np
import pytest

from paper_2609_09020_gb300 import workloads as wk

from test_izpr_gpu import _built  # noqa: F401  (the module's fixture)

pytestmark = pytest.mark.gpu
EOB = 500


def _stream(n, seed):
    """n symbols: literals and single-zero runs, a marker after 0 to 40 of them."""
    rng = np.random.Generator(np.random.PCG64(seed))
    s = rng.integers(-200, 200, n).astype(np.int32)
    s[rng.random(n) < 0.1] = EOB - 16  # a run of one zero
    ends, at = [], -1
    while at < n - 1:
        at = min(at + 1 + int(rng.integers(0, 41)), n - 1)
        ends.append(at)
    s[ends] = EOB
    return s, np.array(ends, np.int64)


SIZES = [(n, k) for n in (1, 3, 2047, 2048, 2049) for k in range(4)]
SIZES += [(n, k) for n in (2048 * 1215 + 5, 2048 * 1216, 2048 * 1217 - 1, 2048 * 3000 + 777) for k in (0, 1)]


@pytest.mark.parametrize("n,skew", SIZES)
def test_ranges(orc, n, skew):
    import torch
    from paper_2609_09020_gb300 import pic
    s, ends = _stream(n, n + skew)
    dev = torch.from_numpy(np.r_[np.full(skew, EOB, np.int32), s]).cuda()[skew:]
    c, o = pic.izpr_decode(dev, EOB, ends.size)
    assert np.array_equal(o.cpu().numpy(), ends)
    assert np.array_equal(c.cpu().numpy(), orc.izpr(s, EOB, ends.size))

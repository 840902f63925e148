"""The order of the row-marching tcgen05 kernel's MMAs on tensor memory,
restated on the CPU.

Two MMAs of one thread run in issue order only if they share accumulator and
shape.  Any other pair that touches the same columns, one of them writing,
needs the first one's completion (a commit that the issuing warp has seen,
itself or through a warp that arrived afterwards) before the second is issued.
The schedule of one group: layer 0 of a tile into a region, each later layer
from that region into the other one, the next tile's layer 0 into the region
that the last layer read.  Whether the issuing warp waits for the last layer
before that is taken from the source.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09020_gb300", "csrc",
                   "k_tcmarch.cuh")


def schedule(layers, tiles, waits_for_last):
    """MMAs of one group as (reads, writes, shape, index of the last MMA known complete)."""
    ops, reg, done = [], 0, -1

    def layer(reads, writes, shape):
        ops.append((reads, writes, shape, done))

    for t in range(tiles):
        if t and waits_for_last:
            done = len(ops) - 1
        layer(None, reg, (128, 64))  # layer 0: operand from shared memory
        for k in range(1, layers):
            done = len(ops) - 1  # the decoding warps have seen the layer before complete
            layer(reg, reg ^ 1, (128, 16 if k == layers - 1 else 64))
            reg ^= 1
        reg ^= 1
    return ops


def unordered(ops):
    for j, (rj, wj, sj, done) in enumerate(ops):
        for i, (ri, wi, si, _) in enumerate(ops[:j]):
            if i <= done or (wi == wj and si == sj):
                continue
            if wj in (ri, wi) or wi == rj:
                yield i, j


def test_the_model_sees_the_missing_wait():
    assert list(unordered(schedule(3, 3, False)))


@pytest.mark.parametrize("layers", [3, 4])
def test_every_conflicting_pair_is_ordered(layers):
    waits = re.search(r"if \(ok && i \+ 1 < tiles\) ok = wait\(my_c, [^;]*\) && first_layer\(\);", open(SRC).read())
    assert not list(unordered(schedule(layers, 4, waits is not None)))

"""The short check in front of Decoder.decode_batch and decode lets through
only what the full check passes: every fault in each of the four buffers, and
arrays that are no tensors, go to the full check."""
import itertools

import numpy as np
import pytest

from paper_2609_09020_gb300 import pic

NEED = {"latents": 64, "steps": 8, "weights": 40, "out": 48}


class _Cuda:
    """What both checks ask of a CUDA tensor."""

    class _Dev:
        def __init__(self, index):
            self.index = index

    def __init__(self, nbytes, index=0, contig=True):
        self.nbytes, self.is_cuda, self.device = nbytes, index >= 0, self._Dev(index)
        self._contig = contig

    def get_device(self):
        return self.device.index

    def is_contiguous(self):
        return self._contig

    def numel(self):
        return self.nbytes

    def element_size(self):
        return 1


def _passes(need, device, bufs):
    try:
        pic.check_decode_buffers(need, 1, 2, 2, device=device, **bufs)
    except ValueError:
        return False
    return True


def test_agrees_with_the_full_check():
    kinds = [lambda n: _Cuda(n), lambda n: _Cuda(n + 3), lambda n: _Cuda(n - 1), lambda n: _Cuda(n, 1),
             lambda n: _Cuda(n, -1), lambda n: _Cuda(n, contig=False), lambda n: None,
             lambda n: np.zeros(n, np.uint8)]
    passed = 0
    for need in (NEED, {**NEED, "steps": 0}):
        for pick in itertools.product(kinds, repeat=4):
            bufs = {k: f(need[k]) for k, f in zip(NEED, pick)}
            fits = pic._buffers_fit(need, 0, **bufs)
            assert fits == _passes(need, 0, bufs), {k: vars(v) if v is not None and hasattr(v, "__dict__") else v
                                                    for k, v in bufs.items()}
            passed += fits
    assert passed


def test_cpu_tensors_go_to_the_full_check():
    torch = pytest.importorskip("torch")
    t = {k: torch.zeros(n, dtype=torch.uint8) for k, n in NEED.items()}
    assert not pic._buffers_fit(NEED, 0, **t)

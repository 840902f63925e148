"""Host state that all calls share (what is looked up once per device) may be
written by several threads on their first calls, so it is atomic or guarded by
a mutex: no plain function-local static in the CUDA sources."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09020_gb300", "csrc")


def test_function_local_statics_are_atomic_or_constant():
    plain = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for line in open(path):
            m = re.match(r"\s+static (?!const\b|constexpr\b|std::atomic<)(.*)$", line)
            if m and "(" not in m.group(1).split("=")[0].split(";")[0]:
                plain.append((os.path.basename(path), m.group(1)))
    assert not plain

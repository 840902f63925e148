"""A CTA's shared memory belongs to the next CTA as soon as it exits, so a
kernel that stages with asynchronous copies waits for the last of them after
its work loop.  Checked in the sources, since a copy that lands late cannot be
provoked: the text between the work loop's end and the end of the role that
issues the copies has the wait."""
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09020_gb300", "csrc")


def _block(text, at):
    """End of the brace block that opens at or after `at`."""
    i, depth = text.index("{", at), 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced braces")


# file, kernel, start of the role that issues the copies
ROLES = [
    ("k_strip.cuh", "strip_decode_kernel(const DecodeParams p)", None),
    ("k_tcmarch.cuh", "march_decode_kernel(const DecodeParams p)", "else if (warp < kDecWarps + kFeatWarps)"),
]


@pytest.mark.parametrize("name,kernel,role", ROLES, ids=[r[0] for r in ROLES])
def test_last_copies_are_waited_for(name, kernel, role):
    text = open(os.path.join(CSRC, name)).read()
    at = text.index(kernel)
    if role:
        at = text.index(role, at)
    body = text[at:_block(text, at)]
    loop = body.index("for (long long seg")
    rest = body[_block(body, loop):]
    assert "features(" in body[loop:_block(body, loop)]
    assert "cp_async_wait_all()" in rest, f"{name}: copies may be in flight when the CTA exits"

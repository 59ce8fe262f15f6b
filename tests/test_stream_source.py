"""Rules of the streaming apply kernel that a run on a GPU cannot be made to break on purpose: the order of its exchange, and what it
does after a wait has run out.  Checked on the source text (no GPU)."""
import os
import re

import pytest

import paper_2603_15965_b200 as M

SOURCE = os.path.join(os.path.dirname(M.__file__), "csrc", "apply_stream.cu")


@pytest.fixture(scope="module")
def code():
    with open(SOURCE) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_slot_is_written_only_after_the_peers_have_read_the_copies_made_from_it(code):
    """A CTA's slot of item i - 2 is the source of asynchronous copies to the peers; the only proof that they are done is the peers'
    arrival on tfree_s, so that wait and a barrier of all compute warps come before item i's partial is written there."""
    shrink = code[code.index("auto shrink = "):code.index("auto expand = ")]
    wait = shrink.index("tfree_s[i & 1]")
    barrier = shrink.index("fs_compute_sync()", wait)
    write = shrink.index("slot_of(i, crank)")
    push = shrink.index("bulk_copy_to_peer(")
    assert wait < barrier < write < push
    assert shrink.count("tfree_s") == 1

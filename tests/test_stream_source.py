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


def test_nothing_is_stored_to_y_after_a_time_out(code):
    """Every wait falls through once one has run out; what the stages and t hold from then on must not reach y."""
    expand = code[code.index("auto expand = "):code.index("shrink(next, i + 1)")]
    # rank 64, where the compute warps store: t is checked once an item, the stage once a chunk
    live = expand.index("live = *static_cast<volatile int*>(&abort_s) == 0")
    leave = expand.index("if (Cfg::DIRECT && !arrived) break;")
    assert expand.index("tfull_s[i & 1]") < live < expand.index("arrived = wait_bar(smem_u32(&full_s[s])") < leave < expand.index("stg128(")
    assert re.search(r"yrow\[mt\]\[h\] = live && row < it.rows \?", expand) and re.search(r"if \(yrow\[mt\]\[h\] != nullptr\)\s*stg128\(", expand)
    assert expand.count("stg128(") == code.count("stg128(") == 1
    # ranks 16 and 32, where the copy warps do
    retire = code[code.index("auto retire = "):code.index("auto token_of = ")]
    assert re.search(r"nb != 0 && !abort_s", retire) and code.count("bulk_store(") == retire.count("bulk_store(") == 1


def test_no_cta_leaves_after_a_time_out_while_copies_between_ctas_may_be_in_flight(code):
    """A CTA that has given up waits for nothing, so the copies to and from it are not known to be done when it reaches the end: the
    whole cluster learns of the time-out, stops at a barrier, lets them land and leaves together."""
    end = code[code.index("expand(cur, i)"):code.index("bool stream_eligible(")]
    tell = end.index("st_cluster_u32(map_to_cta(smem_u32(&abort_s), lane), 1u)")
    stop = end.index("cluster_sync_all()")
    land = end.index("kFsLandingCycles")
    leave = end.index("cluster_sync_all()", land)
    assert tell < stop < land < leave
    assert re.search(r"if \(\*aborted\) \{[^{}]*kFsLandingCycles\) \{\s*\}[^{}]*cluster_sync_all\(\);\s*\}", end)

"""How kernels end after a wait that ran out (checked on the source: nothing makes a wait of these
kernels run out on a GPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_04526_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_adapter_gradient_gives_up_as_a_block():
    """A bounded wait can run out for some of a block's threads only. The adapter gradient's steps
    have block barriers and elections of whole warps, which wait without a limit for threads that
    left: its loop may end on the block's vote alone."""
    src = _source("sq_adapter_tc.cu")
    loop = src[src.index("for (int s = 0; s < steps; ++s)"):src.index("if (ok && dB_all")]
    exits = re.findall(r"if \(([^;{}]*)\) (?:break|return);", loop)
    assert exits == ["!ok"], exits
    assert re.search(r"ok = __syncthreads_and\(ok\);\s*if \(!ok\) break;", loop)


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_commits_come_from_the_lane_that_issued(name):
    """tcgen05.commit waits for the MMAs of the thread that executes it. Where an elected lane
    issues them, a commit by a fixed thread (before TMEM is freed, say) need not wait for any."""
    src = _source(name)
    if "umma_bf16_elect(" in src:
        assert not re.findall(r"\bumma_commit\(", src)
        assert "umma_commit_elect(" in src


def test_aborted_copies_are_waited_for():
    """After an abort every copy in flight is waited for, ring by ring: in the few-token kernel the
    codes (slots) and the activations (stages). A block that ends before a copy lands lets it write
    into the next block's shared memory."""
    src = re.sub(r"\s+", " ", _source("sq_few.cu"))
    for call in ("drain_ring(cfull, j, p.slots)", "drain_ring(full, it, S)"):
        assert f"if (*abort_flag) {call};" in src, call
    assert ("for (int i = (fills > slots ? fills - slots : 0); i < fills; ++i) "
            "mbar_drain(&full[i % slots], static_cast<uint32_t>(i / slots) & 1u);") in src

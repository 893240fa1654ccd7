"""A CTA that gives up on a bulk copy still waits for its copies in flight, by
the full limit and not by the one that fault injection lowers: the shared
memory that they write is another CTA's once it has left."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1402_3281_gb300", "csrc")


def test_copies_in_flight_are_waited_for_by_the_full_limit():
    src = open(os.path.join(CSRC, "lp.cu")).read()
    blocks = re.findall(r"if \(__syncthreads_or\(!ok\)\) \{(.*?)return;", src, re.S)
    assert blocks
    for b in blocks:
        waits = re.findall(r"mbar_wait\([^;]*?,\s*([A-Za-z_.]+)\);", b)
        assert waits == ["WAIT_LIMIT", "WAIT_LIMIT"]

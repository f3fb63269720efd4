"""The cluster masking kernel stores into the other CTAs' shared memory, which
is defined only once they have started. A start that comes late cannot be
brought about on a GPU, so the order is checked in the source: every CTA
arrives at a cluster barrier on entry and waits for it before its first pass,
and all remote stores lie in the passes' sums."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_cta_has_started_before_the_first_remote_store():
    with open(os.path.join(ROOT, "paper_2512_16278_gb300", "csrc", "flag.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = text[text.index("flag_cluster_kernel(FlagArgs f"):]
    body = body[:body.index("\n}\n")]
    sums = body.index("auto cluster3")
    end = body.index("};", sums)
    stores = [m.start() for m in re.finditer(r"\bcl_store\(", body)]
    assert stores and all(sums < at < end for at in stores)
    first = body.index("cluster3(", end)
    arrive, wait = body.index("if (G > 1) cl_arrive();"), body.rindex("if (G > 1) cl_wait();", 0, first)
    assert arrive < sums and end < wait < first

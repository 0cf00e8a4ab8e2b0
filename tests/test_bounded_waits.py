"""Bounded waits in the kernels, by their source: no GPU case can make one of them run out (they are limited to
seconds) without a hang, so what follows a wait that did is looked at here."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_08152_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"\s+", " ", re.sub(r"//[^\n]*", "", text))


def test_prefill_reports_each_wait_that_ran_out():
    src = _source("prefill.cu")
    # a wait whose result is dropped: only those for a role's own copies in flight, as it ends
    dropped = re.findall(r"[;{}] (?:\([a-z]+\) ?)?((?:pf_wait|uni_wait|warp_wait|item_wait)\([^;]*\));", src)
    assert dropped == ["pf_wait(&full[st], ph ^ 1, limit_ns)"], dropped
    # with 64 keys a tile warp_wait leaves its verdict in got_all: it is looked at before every O is stored, the
    # last item's among them, whose pass leaves the loop before the end of a tile
    calls = [m.start() for m in re.finditer(r" epilogue\(", src)]
    assert len(calls) == 1, calls
    assert src[:calls[0]].rstrip().endswith("if (KT == 64 && !(ok = __all_sync(0xFFFFFFFFu, got_all))) break;")

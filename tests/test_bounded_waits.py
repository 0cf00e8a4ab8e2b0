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


def test_decode_lanes_agree_on_a_wait_and_a_dead_part_is_not_merged():
    src = _source("kernels.cu")
    # every wait whose verdict guards warp-wide work is voted on; the others are one lane's, or a role's last
    for wait in re.finditer(r"mbar_wait_bounded\(&full\[stage\]", src):
        assert src[:wait.start()].endswith("__all_sync(kFull, "), src[wait.start() - 80:wait.end() + 60]
    cta = src[src.index("decode_cta_kernel("):]
    # a warp's result carries the verdict, a merge keeps the worst one, and the last merge stores none but good ones
    assert "so[2] = dead ? 1.f : 0.f;" in cta
    assert "bad = fmaxf(bad, sp[w * C::PO + 2]);" in cta
    assert "st_cluster_f32(dst + 2, 0, bad);" in cta
    stores = re.findall(r"if \(([^;{}]*)\) orow\[", cta)
    assert stores and all("bad == 0.f" in s for s in stores), stores

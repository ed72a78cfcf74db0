"""The barrier words of the whitening components spread over several CTAs carry
two sums and the barrier's number.  A reader takes the sums because it sees the
number, so a word must be read and written by one access: a PTX vector access is
several scalar ones in no stated order.  Checked on the source."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_12117_gb300", "csrc",
                   "k_solve.cu")


def _body(name):
    text = open(SRC).read()
    start = text.index(name + "(")
    return text[start:text.index("\n}\n", start)]


def test_barrier_words_are_single_accesses():
    for fn, op in (("ld_slot", "ld"), ("st_slot", "st")):
        accesses = re.findall(r"(?:ld|st|atom|red)\.[\w.]+", _body(fn))
        assert accesses == [f"{op}.relaxed.gpu.global.b128"], (fn, accesses)

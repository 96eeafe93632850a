"""CPU: the grid barrier's accesses to its word.

The memory model orders a release and an acquire only if the two accesses overlap completely, which a
run cannot show: a mixed-width pair passes every test on hardware that reads the word at once.  So the
source is held to it."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_05610_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_every_access_to_the_barrier_word_has_its_width():
    text = code("lf2_barrier.cuh")
    ops = re.findall(r"\b(?:red|atom|ld|st)\.[\w.]*?\.[bu](\d+)\b[^\"]*\[", text)
    assert len(ops) >= 2 and set(ops) == {"64"}, ops
    assert not re.search(r"\batomic[A-Z]\w*\s*\(|\bvolatile\s+unsigned", text)
    assert re.search(r"red\.release\.gpu\.global\.add\.u64", text) and re.search(r"ld\.acquire\.gpu\.global\.u64", text)
    for fn in ("grid_arrive", "grid_wait"):
        assert re.search(fn + r"\(unsigned long long \*bar\b", text), fn

"""The grid barrier's word: a release, a relaxed read and the fence after it
order two blocks' accesses only where all accesses to the word have one size
(PTX memory model, morally strong operations), so every one of them is of 64
bits -- arrivals, polls and the error bit."""
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2411_16667_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _body(text, head):
    """The text of the block that follows head."""
    a = text.index("{", text.index(head))
    depth, b = 0, a
    while True:
        depth += {"{": 1, "}": -1}.get(text[b], 0)
        b += 1
        if depth == 0:
            return text[a:b]


def test_every_access_to_the_barrier_word_is_of_64_bits():
    dev = _source("opmos_dev.cuh")
    fields = dict(reversed(f.split()) if len(f.split()) == 2 else (f.split()[-1], " ".join(f.split()[:-1]))
                  for f in _body(dev, "struct alignas(16) Barrier").strip("{}").split(";") if f.strip())
    assert fields["state"] == "unsigned long long" and fields["error"] == "unsigned"
    wait = _body(dev, "bool grid_barrier(Barrier*")
    ops = re.findall(r'asm volatile\("(\S+) ([^"]*)"(.*?)\);', wait, re.S)
    assert [op.split(".")[0] for op, _, _ in ops] == ["red", "ld"]
    for op, _, operands in ops:
        assert op.endswith(".u64") and "&b->state" in operands and "error" not in operands
    assert "atomicOr(&b->state, kBarError)" in _body(dev, "void set_error(Barrier*")
    # nothing else touches the word, and the bit is set after the code is written
    uses = sum(len(re.findall(r"\bstate\b", _body(dev, f))) for f in ("bool grid_barrier(Barrier*", "void set_error(Barrier*"))
    assert len(re.findall(r"(?:->|\.)state\b", dev)) == uses
    setter = _body(dev, "void set_error(Barrier*")
    assert setter.index("atomicCAS(&b->error") < setter.index("__threadfence") < setter.index("atomicOr(&b->state")
    for name in os.listdir(CSRC):
        assert not re.search(r"bar(?:->|\.)state\b|atomicCAS\(&\w+->(?:bar\.)?error", _source(name)) or name == "opmos_dev.cuh"

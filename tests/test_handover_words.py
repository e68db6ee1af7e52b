"""The words in which one CTA of a sweep hands results to another (a value with its tag, or a value that says by itself
whether it is there) have 64 bits.  PTX makes only each element of a vector access a single access, so the elements of
every load and store of such words have to be 64 bits long."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_13483_gb300", "csrc")


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def test_strong_global_accesses_move_whole_words():
    found = 0
    for f, text in sources().items():
        for m in re.finditer(r"\b(?:ld|st)\.(?:volatile|relaxed\S*?)\.global((?:\.v[24])?)\.([a-z]\d+)", text):
            found += 1
            assert m.group(2) in ("u64", "b64"), (f, m.group(0))
    assert found >= 4


def test_tagged_words_are_stored_whole():
    text = sources()["ops.cu"]
    assert not re.search(r"\btag\[[^;]*\]\s*=[^=]", text)   # a plain 16-byte store has no element size of its own
    assert len(re.findall(r"\bst_tag\(tag", text)) == 2

"""include/seedq.h says of the error word what sets it: every kernel file that
sets a bit for a wait that ran out has the header mention waits."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_error_word_names_the_bounded_waits():
    csrc = os.path.join(ROOT, "paper_2609_38477_gb300", "csrc")
    waits = [f for f in os.listdir(csrc) if f.endswith((".cu", ".cuh"))
             and re.search(r"if \(!mbar_wait[^{]*\{[^}]*atomicOr\(p\.flags", open(os.path.join(csrc, f)).read(), re.S)]
    assert waits == ["decode.cu"]
    header = open(os.path.join(ROOT, "include", "seedq.h")).read()
    text = header[header.index("Device error flags accumulated"):header.index("seedq_status seedq_last_device_error")]
    assert "full decode" in text and "waits" in text

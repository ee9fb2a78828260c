"""Rules of programmatic dependent launches that hold in the sources: a kernel may be
resident while its predecessor still writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_05260_gb300", "csrc")


def _sources():
    out = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(p) as f:
            out[os.path.basename(p)] = re.sub(r"//[^\n]*", "", f.read())
    return out


def test_no_non_coherent_loads_of_what_kernels_write():
    for name, text in _sources().items():
        assert not re.search(r"ld\.global(\.\w+)*\.nc", text), name
        # the rest tables, which no kernel of a frame writes, are the one exception
        for arg in re.findall(r"__ldg\(([^;]*?)[,)]", text):
            assert arg.startswith("RV2"), (name, arg)


def test_kernels_wait_before_they_release_their_successor():
    found = 0
    for name, text in _sources().items():
        for body in re.split(r"\b__global__\b", text)[1:]:
            trigger = body.find("pdl_trigger()")
            if trigger < 0 or "void pdl_trigger" in body:
                continue
            found += 1
            wait = body.find("pdl_wait()")
            assert 0 <= wait < trigger, (name, body[:80])
    assert found >= 10

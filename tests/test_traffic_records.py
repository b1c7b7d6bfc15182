"""The recorded DRAM traffic of a kernel counts only while its sources are the ones
measured: every record names all of the library's files that the kernel is built from."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_10305_gb300", "csrc")


def included(name, seen):
    seen.add(name)
    for inc in re.findall(r'#include "(gpz_\w+\.cuh)"', open(os.path.join(CSRC, name)).read()):
        if inc not in seen:
            included(inc, seen)
    return seen


@pytest.mark.parametrize("kernel,source", [("range", "gpz_qse.cu"), ("qse", "gpz_qse_tile.cu"),
                                           ("compact", "gpz_compact.cu"), ("decompress", "gpz_decode.cu")])
def test_a_record_names_all_its_sources(kernel, source):
    text = open(os.path.join(ROOT, "profiles", "traffic_%s.txt" % kernel)).read()
    assert set(re.findall(r"^sha256 (\S+):", text, re.M)) == included(source, set())

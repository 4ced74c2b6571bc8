"""The library is rebuilt when any file that it is made of has changed."""
import os
import re

from paper_2310_07182_gb300 import build


def test_every_source_file_is_a_build_input():
    files = {f for f in os.listdir(build.CSRC) if re.search(r"\.(cu|cuh|cpp|h)$", f)}
    assert files == set(build.SOURCES) | set(build.HEADERS)

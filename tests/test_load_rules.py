"""A kernel launched programmatically is resident before its source has been written.  What it reads behind its wait it has to read with
coherent loads: the non-coherent path (ld.global.nc, __ldg) asks for data that nobody writes while the kernel runs, and the compiler may
move an __ldg ahead of the wait."""
import os
import re

import pytest

from paper_2509_25149_b200 import build

# The reductions of metrics.cu are no case of it: the kernel that clears their sums has waited for the source before they start.
BEHIND_ZERO_WORDS = {"metrics.cu"}


def without_comments(text):
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


@pytest.mark.parametrize("name", [f for f in build.SOURCES + build.HEADERS if f not in BEHIND_ZERO_WORDS])
def test_sources_are_read_with_coherent_loads(name):
    text = without_comments(open(os.path.join(build.CSRC, name)).read())
    assert not re.findall(r"__ldg\s*\(|ld\.global[\w.:]*\.nc\b", text)

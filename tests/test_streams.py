"""Every device operation of the library is ordered by the context's stream.

That stream does not wait for the legacy default stream, so a fill or a copy
enqueued there is ordered with no kernel that relies on it: the reductions'
tickets, the coarse solver's barrier words and the neighbour table have to be
written on the stream their readers run on.  Read from the sources, so that it is
checked without a GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1509_06865_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) +
               glob.glob(os.path.join(CSRC, "*.h")))


def _code(path):
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


def _span(text, i, opening, closing):
    """The text from the opening bracket at i to its partner."""
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == opening) - (text[j] == closing)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced")


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_device_work_names_the_contexts_stream(path):
    text = _code(path)
    assert not re.findall(r"\bcudaMem(?:cpy|set)(?:2D|3D)?\s*\(", text), "on the default stream"
    for m in re.finditer(r"\bcudaMem(?:cpy|set)\w*Async\s*\(|\bcudaLaunchCooperativeKernel\s*\(", text):
        call = _span(text, m.end() - 1, "(", ")")
        assert re.search(r"\bstream\s*\)$", call), call
    for m in re.finditer(r"<<<(.*?)>>>", text, flags=re.S):
        assert re.search(r",\s*(?:\w+\.)*stream$", m.group(1)), m.group(0)

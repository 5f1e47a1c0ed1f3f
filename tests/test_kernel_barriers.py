"""Named barriers of the kernels, read from the sources: a warp that arrives on a barrier without waiting there may be at the next meeting
before the others have left the first, and its second arrival would stand in for a late warp.  So an id that is only arrived on has one meeting
in its file, and is not 0, which __syncthreads meets on."""
import os
import re

import pytest

from paper_2509_22323_b200 import build


def barrier_calls(text, name):
    return [int(n) for n in re.findall(r"\b%s\((\d+)," % name, re.sub(r"//[^\n]*", "", text))]


@pytest.mark.parametrize("source", build.SOURCES)
def test_a_barrier_arrived_on_without_a_wait_is_met_once(source):
    with open(os.path.join(build.CSRC, source)) as f:
        text = f.read()
    arrived, met = barrier_calls(text, "bar_arrive"), barrier_calls(text, "bar_sync")
    assert len(re.findall(r"\bbar_(?:arrive|sync)\(", re.sub(r"//[^\n]*", "", text))) == len(arrived) + len(met)   # all with an id in numbers
    for i in arrived:
        assert i != 0, "__syncthreads meets on 0"
        assert arrived.count(i) == 1 and met.count(i) == 1

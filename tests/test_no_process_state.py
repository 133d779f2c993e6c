"""Kernel choices belong to a context (its device): the files of the visits, the split sweeps, the
prolongation and the bottom keep no variable for the whole process, which the last context created would
set for all others."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1511_08200_gb300", "csrc")


@pytest.mark.parametrize("name", ["k_visit.cu", "k_split.cu", "k_prolong.cu", "k_bottom.cu"])
def test_no_variable_at_namespace_scope(name):
    text = open(os.path.join(CSRC, name)).read()
    found = [line for line in text.splitlines()
             if re.match(r"(static |inline |thread_local |std::)*[\w:<>]+ \w+( = [^;()]*)?;", line)
             and not re.match(r"(using|template|struct|class|return|namespace|constexpr|static constexpr) ", line)]
    assert not found, found

"""Kernels launched with programmatic stream serialization live while the kernels before them still write: in the sources
whose kernels are all launched that way, no load may claim that memory is read-only for the kernel's lifetime."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09821_b200", "csrc")


@pytest.mark.parametrize("name", ["update.cu", "ppo.cu", "mlp_simt.cu", "mlp_tc.cu"])
def test_no_read_only_loads(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "launch_pdl(" in text and "__ldg(" not in text and "ld.global.nc" not in text
    assert not re.search(r"const \w+ \*__restrict__", text)            # (the compiler may make such loads of them)

"""Kernels that start under the stream's previous kernel read what that kernel may have written through coherent loads
only: in their sources nothing but the twiddle tables, fixed since they were made, is marked for the read-only path."""

import os
import re

import pytest

from paper_2605_28451_gb300 import build

CHAINED = [f for f in sorted(os.listdir(build.CSRC))
           if "chain_begin();" in open(os.path.join(build.CSRC, f)).read() and f != "async_copy.cuh"]


def test_the_kernels_are_found():
    assert {"fft_rows.cuh", "wide_rows.cuh", "long_rows.cuh", "tc_fft.cuh", "transpose.cu", "rda.cu"} <= set(CHAINED)


@pytest.mark.parametrize("name", CHAINED)
def test_only_tables_are_read_as_constant(name):
    text = re.sub(r"//.*", "", open(os.path.join(build.CSRC, name)).read())
    marked = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", text)
    loaded = re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([\w.]+)", text)
    assert all(re.fullmatch(r"tw\w*", v) for v in marked), marked
    assert all(re.fullmatch(r"(a\.)?tw\w*|row", v) for v in loaded), loaded     # row: of the table, in wide_rows.cuh

"""Kernels that are launched while their predecessor still runs must not read what it writes through the read-only
data path (const __restrict__ parameters, __ldg), which wants memory that does not change in a kernel's whole life."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_10389_b200", "csrc")
SOURCES = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cuh", ".cu"))}
ALL = "\n".join(SOURCES.values())


# kernel, parameter: a chain's first kernels read the caller's buffers; the others what the chain has written
@pytest.mark.parametrize("kernel,parameter", [("k_chunk_crcs", "cache"), ("k_encode_init", "dirty"), ("k_decode_check", "wire"),
                                              ("k_diff_compact", "dirty"), ("k_decode_finish", "dst"), ("describe_tile", "plist")])
def test_parameters_a_predecessor_may_still_write_are_plain_pointers(kernel, parameter):
    signature = re.search(r"\b%s\(((?:[^()]|\([^()]*\))*)\)\s*\{" % kernel, ALL).group(1)
    declared = [p for p in signature.split(",") if re.search(r"\b%s$" % parameter, p.strip())]
    assert len(declared) == 1 and "__restrict__" not in declared[0]


def test_the_workspace_is_not_read_through_the_read_only_path():
    for name, text in SOURCES.items():
        assert not re.search(r"__ldg\(\s*&?ws\.", text), name

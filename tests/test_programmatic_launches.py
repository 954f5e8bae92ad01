"""The rules of programmatic dependent launches, checked on the kernels' source:
a dependent is resident while the kernel before it still runs.
"""
import os
import re

from paper_2608_26004_gb300.build import CSRC


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", text)  # (comments aside)


def test_what_the_map_check_writes_is_not_read_as_read_only():
    # fuse_verify_xrow is resident while xvocab_inv_build writes the inverse map
    # and the error word: read-only (non-coherent) loads of them are undefined
    text = source("kernel_xrow.cuh")
    reads = re.findall(r"(\w+)\(\s*(?:reinterpret_cast<[^>]*>\()?\s*X\.(inv_v|map_err)", text)
    assert {what for _, what in reads} == {"inv_v", "map_err"}
    assert all(load == "__ldcg" for load, _ in reads), reads
    assert len(reads) == len(re.findall(r"X\.(?:inv_v|map_err)\b", text))

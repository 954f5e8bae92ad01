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


def test_every_programmatic_dependent_waits():
    # a kernel launched with the attribute executes griddepcontrol.wait on every
    # path that ends it (the wait may lie in a function it calls)
    host = source("asymspec.cu")
    assert host.count("programmaticStreamSerializationAllowed = 1") == 3
    for name, kernel in (("kernel_tma.cuh", "decide_rows"), ("kernel_row.cuh", "decide_element"),
                         ("kernel_full.cuh", "decide_full"), ("kernel_xrow.cuh", "fuse_verify_xrow"),
                         ("kernel_xvocab.cuh", "xvocab_gather_inv")):
        text = source(name)
        body = text[text.index(" " + kernel + "("):].split("\ntemplate")[0]
        first = re.search(r"griddepcontrol\.wait|\breturn;", body)
        assert first and first.group().startswith("griddep"), kernel
    # (the gather waits in its last CTA, through a lambda called before each exit)
    body = source("kernel_xvocab.cuh").split(" xvocab_gather_inv(")[1].split("\ntemplate")[0]
    assert len(re.findall(r"wait_for_gather\(\);\s*(?:return;|\})", body)) == 2
    assert len(re.findall(r"\breturn;", body)) == 1

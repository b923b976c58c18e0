"""Kernels that wait for the kernel before them read what it has written: a pointer that read-only loads go through has to come out
of grid_wait(), or nothing orders those loads behind the wait (they have no order of their own against it)."""
import glob
import os
import re

import pytest

from paper_2605_06665_b200 import build as builder


def kernels():
    """(file:kernel, (its body, the names declared as pointers in its file)) of every kernel."""
    for path in sorted(glob.glob(os.path.join(builder.CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?:[^(){}]|\([^()]*\))*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield f"{os.path.basename(path)}:{m.group(1)}", (text[m.end():i], set(re.findall(r"\*\s*(\w+)\s*[;,]", text)))


ALL = dict(kernels())


def test_all_kernels_are_seen():
    assert len(ALL) >= 20 and {"route_few.cu:route_few_kernel", "expert_simt.cu:grouped_rows_gemm_kernel",
                               "dispatch.cu:combine_kernel"} <= set(ALL)


@pytest.mark.parametrize("name", sorted(ALL))
def test_pointers_of_read_only_loads_come_out_of_the_wait(name):
    body, pointers = ALL[name]
    if "grid_wait" not in body or not re.search(r"\b(__ldg|ld4)\(", body):
        return
    waited = set(re.findall(r"[\w.]+", re.search(r"grid_wait\(([^)]*)\)", body).group(1)))
    # pointers in a parameter struct that addresses are formed from, but for those that are written through
    read = {n for n in re.findall(r"\bp\.(\w+)(?= \+)", body) if n in pointers}
    read -= {n for n in read if re.search(rf"(st4|atomic\w+)\(&?p\.{n}\b", body)} | {"dW", "f"}   # dW: in place, plain loads; f: a width
    read = {"p." + n for n in read}
    assert waited and read <= waited, (read, waited)

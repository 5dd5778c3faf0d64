"""Kernels that are launched while the one before runs read global memory by ordinary loads.

The read-only path (__ldg, const __restrict__ parameters) wants data that nobody writes while the kernel runs.  A kernel that
is launched early runs while the one before still writes its operands, so a line that an SM has in its cache from an older
reader may be the old one.  No run shows that reliably; the sources do.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_05350_b200", "csrc")


def sources():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            yield name, re.sub(r"//[^\n]*", "", f.read())


def launched_early(text):
    return re.search(r"\blaunch_k(_if)?\(|ProgrammaticStreamSerialization", text) is not None


@pytest.mark.parametrize("name,text", [(n, t) for n, t in sources() if n.endswith(".cu") and launched_early(t)], ids=lambda v: v if v.endswith(".cu") else "")
def test_a_kernel_launched_early_reads_by_ordinary_loads(name, text):
    assert "__ldg" not in text
    assert re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+\w+", text) == []
    # the read-only path for what a model holds: only in the kernel that runs whole models
    assert name == "chain_cluster.cu" or "load_fixed" not in text


def test_headers_read_by_ordinary_loads():
    for name, text in sources():
        if name.endswith(".cuh"):
            assert text.count("__ldg") == (1 if name == "common.cuh" else 0), name  # load_fixed itself
            assert re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+\w+", text) == [], name


def test_kernels_that_read_through_the_read_only_path_are_launched_after_the_one_before():
    """The others: no launch in their files carries the attribute."""
    others = [n for n, t in sources() if n.endswith(".cu") and ("__ldg" in t or re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", t))]
    assert others == ["bf16_storage.cu", "conv2d_fp32_simt.cu", "gemm_fp32_simt.cu"]

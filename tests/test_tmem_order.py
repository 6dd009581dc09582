"""Order of tensor-memory stores behind the MMAs that read the same columns, by
reading the CUDA sources (no GPU): a pipeline's decoders and converters store
operands (tcgen05.st) to columns that earlier asynchronous MMAs have read.  The
mbarrier wait that says those MMAs are done orders the stores only together
with a tcgen05.fence::after_thread_sync between the wait and the store."""
import glob
import os
import re

import pytest

from conftest import ROOT

SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2607_16973_gb300", "csrc", "*.cu")))
STORE = re.compile(r"\b(\w*st(?:16|32))\(")         # the tcgen05.st helpers (definitions left out below)
WAIT = re.compile(r"\b(?:warp|all|mbar)_wait\(")
FENCE = re.compile(r"\btc_fence_after\(\)")


def _helpers(text):
    """Names of the functions whose body is a tcgen05.st."""
    return set(re.findall(r"void (\w+)\(.*\) \{\s*asm volatile\(\s*\"tcgen05\.st\.", text))


def _stores(path):
    with open(path) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    names = _helpers(text)
    for m in STORE.finditer(text):
        if m.group(1) in names and not text[:m.start()].rstrip().endswith("void"):
            waits, fences = ([x.start() for x in p.finditer(text, 0, m.start())] for p in (WAIT, FENCE))
            yield text.count("\n", 0, m.start()) + 1, waits[-1], fences[-1]


def test_the_stores_are_found():
    assert {os.path.basename(p) for p in SOURCES if list(_stores(p))} == \
        {"tq_encode_h.cu", "tq_encode_tc.cu", "tq_scan_tm.cu"}


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_a_fence_follows_the_last_wait_before_a_tensor_memory_store(path):
    for line, wait, fence in _stores(path):
        assert fence > wait, f"{os.path.basename(path)}:{line}: tcgen05.st without a fence behind its wait"

"""Every copy and memset of the library runs on the caller's stream.

A context may be bound to a non-blocking stream, which nothing orders after the legacy
default stream: a ``cudaMemset`` or ``cudaMemcpy`` of device memory may still be pending
there when the first kernel of the context starts.  Checked on the sources.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_5536_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_no_copy_or_memset_on_the_legacy_stream(name):
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert not re.findall(r"\bcuda(?:Memset|Memcpy)(?:2D|3D|ToSymbol|FromSymbol)?\s*\(", code)
    # the asynchronous forms name a stream
    for call in re.findall(r"\bcudaMem(?:set|cpy)Async\s*\(((?:[^()]|\((?:[^()]|\([^()]*\))*\))*)\)", code):
        assert re.search(r"(stream|\bst)\s*$", call.strip()), call


def test_sources_of_copies_to_the_device_outlive_them():
    """A copy enqueued from pageable memory may read it later (the host's page tables are the
    device's on Grace-Blackwell): tables are copied from vectors that the context keeps."""
    with open(os.path.join(CSRC, "dg_capi.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    for src in re.findall(r"cudaMemcpyAsync\(\s*[^,]+,\s*([^,]+?),[^;]*cudaMemcpyHostToDevice", code):
        assert ".data()" not in src or src.startswith("c->"), src

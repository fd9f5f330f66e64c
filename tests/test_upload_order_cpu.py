"""Uploads through the legacy stream are ordered before the kernels of a context's own stream.

A synchronous copy from pageable memory may return once the data is staged, and a fill returns at
once; a context stream created non-blocking does not wait for either. No run shows the race at
will, so the sources are checked: uploads belong on the context's stream, except in the two create
calls, which wait for the legacy stream after the last of theirs."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1607_02560_gb300", "csrc")
UPLOAD = re.compile(r"cudaMemcpy\([^;{]*?cudaMemcpyHostToDevice|cudaMemset\(|cudaMemcpyToSymbol\("
                    r"|(?<![\w ] )\bupload_(?:sym|cls125)\(", re.S)
WAIT = "cudaStreamSynchronize(cudaStreamLegacy)"


def body(name, entry):
    """Text of one function, from its name to the closing brace in the first column."""
    text = open(os.path.join(CSRC, name)).read()
    at = text.index(entry)
    return text[at:text.index("\n}", at)]


@pytest.mark.parametrize("name,entry", [("lsp_api.cu", "lsp_status lsp_create("),
                                        ("k_mlp.cu", "lsp_status lsp_mlp_create(")])
def test_create_waits_for_its_uploads(name, entry):
    text = body(name, entry)
    last = [m.end() for m in UPLOAD.finditer(text)][-1]
    first_launch = text.find("retile(m)")
    assert text.find(WAIT, last) >= 0
    assert first_launch < 0 or text.find(WAIT, last) < first_launch


def test_no_other_function_uploads_through_the_legacy_stream():
    create = {("lsp_api.cu", "lsp_status lsp_create("), ("k_mlp.cu", "lsp_status lsp_mlp_create("),
              ("k_eig.cu", "cudaError_t upload_sym("),
              ("k_eig_dense.cu", "cudaError_t upload_cls125(")}
    for name in sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")):
        text = open(os.path.join(CSRC, name)).read()
        for n, entry in create:
            if n == name:
                text = text.replace(body(name, entry), "")
        assert not UPLOAD.search(text), (name, UPLOAD.search(text).group(0)[:80])

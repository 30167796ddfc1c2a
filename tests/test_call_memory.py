"""Temporary memory of a call is handed back on every way out of it: the sampler and the
spread take theirs through CallBuf, whose destructor frees it, and nothing in them takes or
frees such memory by hand (CPU, from the source text)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_10982_gb300", "csrc")


@pytest.mark.parametrize("name", ["sample.cu", "spread.cu"])
def test_temporaries_have_an_owner(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    assert "CallBuf " in text
    assert not re.findall(r"\b(?:call_alloc|cudaMallocAsync|cudaFreeAsync)\s*\(", text)


def test_the_owner_frees_and_cannot_be_copied():
    text = open(os.path.join(CSRC, "internal.cuh")).read()
    body = text[text.index("class CallBuf {"):]
    body = body[:body.index("\n};")]
    assert re.search(r"~CallBuf\(\) \{\s*if \(p_\) cudaFreeAsync\(p_, st_\);", body)
    assert "CallBuf(const CallBuf &) = delete;" in body and "operator=(const CallBuf &) = delete;" in body

"""Scores and selections read the error of their launches before they wait for them: waiting for
the stream does not report a launch that was refused, and the results of an earlier one would
stand in its place."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01752_gb300", "csrc")


def _body(file, function):
    """Text of a function's definition, comments taken out."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    at = re.search(r"sisso_status " + function + r"\([^;{]*\)\s*\{", text).end()
    depth, end = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return text[at:end]


@pytest.mark.parametrize("file,function", [("pair_tc.cu", "pair_tc_scores"), ("sis.cu", "sis_select")])
def test_launch_errors_are_read_before_waits(file, function):
    body = _body(file, function)
    waits = [m.start() for m in re.finditer("cudaStreamSynchronize", body)]
    last = body.rfind("<<<")
    assert last >= 0
    for w in waits:
        launch = body.rfind("<<<", 0, w)
        assert launch < 0 or "cudaGetLastError" in body[launch:w], body[launch:w]
    assert any(w > last for w in waits) or "cudaGetLastError" in body[last:]

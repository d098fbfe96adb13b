"""Failure paths of the ALNS kernel, by its source: every device-side failure goes
through fail_run (the team's barriers read the flag it raises, not the error
word), and no wait's result is dropped, so that a CTA whose wait ran out leaves
instead of working on what the others have not written.  (Making a wait inside
a step run out on a GPU needs a CTA that stops there, which no entry point can
ask for; tests/test_wait_limit_gpu.py covers the first barrier.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def source():
    with open(os.path.join(ROOT, "paper_2602_23685_gb300", "csrc", "alns.cu")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_failure_raises_the_flag():
    src = source()
    writes = [m.start() for m in re.finditer(r"atomic\w+\(&\s*(?:t\.)?ctl->err\b|ctl->err\s*=[^=]", src)]
    body = re.search(r"void fail_run\(AlnsCtl\* ctl, int why\) \{(.*?)\n\}", src, re.S)
    assert body and "GEN_FAILED" in body.group(1)
    assert writes and all(body.start() < w < body.end() for w in writes), \
        [src[w:w + 60] for w in writes if not body.start() < w < body.end()]


def test_no_wait_result_is_dropped():
    src = source()
    for name in ("await_count", "await_release", "team_wait", "team_barrier_select", "grid_barrier", "phase_matrix"):
        calls = [m.start() for m in re.finditer(r"\b%s\(" % name, src)]
        assert calls, name
        for c in calls:
            before = src[:c].rstrip()
            # a definition ("bool name("), or a use in an expression; a bare statement
            # follows ';', '{', '}' or the ')' of an if
            assert before[-1] not in ";{})", (name, src[c - 80:c + 60])

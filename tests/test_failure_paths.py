"""Failure paths of the ALNS kernel, by its source: every device-side failure goes
through fail_run (the team's barriers read the flag it raises, not the error
word)."""
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

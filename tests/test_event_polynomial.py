"""The event kernel's sin^2(pi r), read from the source: the packed form that the kernel calls carries the
constants of the one-phase form, whose error another test bounds, in the same order, and nothing else."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_15253_gb300", "csrc")


def _constants(src, head):
    body = src[src.index(head):]
    return re.findall(r"-?\d+\.\d+(?:e[-+]?\d+)?f", body[:body.index("\n}\n")])


def test_packed_constants_are_the_checked_ones():
    src = open(os.path.join(CSRC, "dev_model.cuh")).read()
    one = _constants(src, "float sin2pi(float r)")
    assert len(one) == 8
    assert _constants(src, "f32x2 sin2pi2(f32x2 r)") == one
    events = open(os.path.join(CSRC, "events.cu")).read()
    run = events[events.index("void survival_run("):]
    run = run[:run.index("\n}\n")]
    assert "sin2pi2(r)" in run
    assert set(re.findall(r"-?\d+\.\d*f", run)) == {"1.f", "-1.f"}   # no constants of its own

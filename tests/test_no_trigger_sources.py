"""No kernel lets its successor in before its own CTAs exit: programmatic launch serialisation
without a trigger (a trigger was measured slower, and a kernel that raised one would have to be
proved safe for every kernel that may follow it). A source check, comments left out; no GPU."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_04245_gb300", "csrc")
TRIGGER = re.compile(r"griddepcontrol\.launch_dependents|cudaTriggerProgrammaticLaunchCompletion|\bpdl_trigger\b")


def _code(text):
    """The text without // and /* */ comments (string literals, which hold PTX, are kept)."""
    return re.sub(r'//[^\n]*|/\*.*?\*/|("(?:\\.|[^"\\\n])*")', lambda m: m.group(1) or "", text, flags=re.S)


def test_comments_are_left_out_and_strings_kept():
    t = 'a; // griddepcontrol.launch_dependents\nasm("griddepcontrol.launch_dependents;"); /* pdl_trigger() */'
    assert len(TRIGGER.findall(t)) == 3 and TRIGGER.findall(_code(t)) == ["griddepcontrol.launch_dependents"]


def test_no_kernel_triggers():
    files = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".cpp"))]
    assert len(files) > 10
    for f in files:
        assert not TRIGGER.search(_code(open(os.path.join(CSRC, f)).read())), f

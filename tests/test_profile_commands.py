"""Every ncu capture command that the profile notes record leaves the clocks
of the GPU alone (--clock-control none): the notes are there to be repeated,
on machines that are shared."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def captures(text):
    """The ncu command lines of a note: whole lines of a fenced block
    (continued by a backslash) and inline code spans."""
    parts = text.split("```")
    for block in parts[1::2]:
        for line in re.sub(r"\\\n\s*", " ", block).split("\n"):
            m = re.search(r"(?:^|&&|;)\s*(ncu\s.*)", line)
            if m:
                yield m.group(1)
    for prose in parts[0::2]:
        for span in re.findall(r"`([^`]+)`", prose):
            if re.match(r"ncu\s+-", span):
                yield " ".join(span.split())


@pytest.mark.parametrize("note", sorted(glob.glob(os.path.join(ROOT, "profiles", "*.md"))), ids=os.path.basename)
def test_captures_leave_the_clocks_alone(note):
    with open(note) as f:
        found = [c for c in captures(f.read()) if not re.match(r"ncu\s+(-i|--import|--list)", c)]
    for c in found:
        assert "--clock-control none" in c, c

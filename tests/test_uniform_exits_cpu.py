"""An error word that another CTA may write at any moment is read by one thread,
which decides for its CTA (or cluster): threads that each read it could leave a
loop one by one while the rest wait for them at a barrier without a limit."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2402_15253_gb300", "csrc")


def reads(name):
    """(line number, line, the innermost enclosing `if` of one thread) of every
    status_of call in a source file, comments removed."""
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"//[^\n]*", "", text)
    out, stack, pending = [], [], ""
    for no, line in enumerate(text.split("\n"), 1):
        if "status_of(" in line:
            out.append((no, line.strip(), [s for s in stack if s]))
        for ch in line:
            if ch == "{":
                stack.append(pending.strip())
                pending = ""
            elif ch == "}":
                stack.pop()
                pending = ""
            elif ch == ";":
                pending = ""
            else:
                pending += ch
        pending += " "
    return out


ONE_THREAD = re.compile(r"if \(.*(threadIdx\.x == 0|lane == 0).*\)$")


@pytest.mark.parametrize("name", ["batched.cu", "peelone.cuh"])
def test_one_thread_reads_the_status(name):
    found = reads(name)
    assert found
    for no, line, scopes in found:
        assert any(ONE_THREAD.search(s) for s in scopes), f"{name}:{no}: {line}"

"""How the launchers raise a kernel's shared-memory limit, read from their sources (one GPU cannot show it): the limit
belongs to the device that is current, so no launcher may raise it once per process only; and it is shared by the
threads that launch the kernel, so it is one bound for every call, not the size that this call needs."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_21627_gb300", "csrc")


def _launchers():
    """(file, body) of every function that calls cudaFuncSetAttribute; bodies start at the last line that begins in
    column 0 and ends with an opening brace."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaFuncSetAttribute\(", src):
            start = [f.start() for f in re.finditer(r"^\S[^\n;]*(?:\n[^\n;{}]*)?\{$", src[:m.start()], flags=re.M)][-1]
            end = src.find("\n}", m.start())
            yield os.path.basename(path), src[start:end]


LAUNCHERS = list(_launchers())


def test_launchers_are_found():
    assert len(LAUNCHERS) >= 8


@pytest.mark.parametrize("i", range(len(LAUNCHERS)))
def test_the_limit_is_raised_on_every_launch(i):
    name, body = LAUNCHERS[i]
    assert not re.search(r"\bstatic\s+(const\s+)?\w+(\s+\w+|\s*<[^>]*>\s*\w+)\s*[=;{]", body), f"{name}: kept between calls:\n{body}"


@pytest.mark.parametrize("i", range(len(LAUNCHERS)))
def test_the_limit_is_the_same_in_every_call(i):
    name, body = LAUNCHERS[i]
    for call in re.findall(r"cudaFuncSetAttribute\((?:[^()]|\([^()]*\))*\)", body):
        limit = call.split("cudaFuncAttributeMaxDynamicSharedMemorySize,")[1]
        assert not re.search(r"\bsmem\b", limit), f"{name}: {call}"

"""Kernels launched before the one ahead of them in the stream has finished
(launch_early) wait for it before they read, and read with ordinary loads: the
read-only path takes memory that does not change while the kernel runs."""

import glob
import os
import re

import pytest

from paper_2607_13205_gb300.build import CSRC


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_no_read_only_loads(path):
    assert not re.findall(r"__ldg\w*|ld\.global\.nc\S*|__restrict__|__restrict\b", _code(path))


def test_early_kernels_wait_first():
    code = {f: _code(f) for f in FILES}
    launched = set()
    for c in code.values():
        for arg in re.findall(r"launch_early\((\w+)", c):
            # a local pointer: the kernels it may stand for
            named = re.findall(rf"auto\* {arg} = (.*?);", c, flags=re.S)
            launched |= set(re.findall(r"\w+_kernel", " ".join(named) if named else arg))
    assert launched >= {"select_kernel", "maxpool_kernel", "snapkv_lse_kernel", "quest_kernel", "compact_kernel",
                        "decode_partial_kernel", "decode_combine_kernel"}
    for k in launched:
        body = next(c[m.end():] for c in code.values() for m in [re.search(rf"\b{k}\(const", c)] if m)
        before = body[body.index("{"):body.index("wait_for_previous_kernels()")]
        # no exit and no access to a tensor (through the arguments) before the wait
        assert "return" not in before and "__global__" not in before
        assert not re.search(r"\ba\.\w+\s*\[", before)

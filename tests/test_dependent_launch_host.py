"""Kernels launched to overlap the one before them (programmatic dependent launch)
touch no memory before they wait for it: whatever stands before pdl_wait() in a
kernel's body declares, and neither reads nor writes."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2305_05055_gb300", "csrc")
DECLARES = re.compile(r"^(extern )?__shared__ [^=]*$|^constexpr |^static_assert\(|^typedef "
                      r"|^\w[\w:<>, ]*& \w+ = (\*reinterpret_cast<|\w+\.\w+$)")


def kernels(text):
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__\s+void[^;{]*?\b(k_\w+)\([^{;]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("unit", ["cpma.cu", "scan.cu", "sort.cu", "update.cu", "query.cu"])
def test_nothing_but_declarations_before_the_wait(unit):
    seen = 0
    for name, body in kernels(open(os.path.join(SRC, unit)).read()):
        if "pdl_wait();" not in body:
            continue
        seen += 1
        for s in body.split("pdl_wait();")[0].split(";"):
            s = " ".join(s.split())
            assert not s or DECLARES.match(s), (name, s)
    assert seen

"""The rule of programmatic dependent launch, read from the sources: until a kernel's own griddepcontrol.wait nothing vouches
for what earlier kernels wrote, so no input is read before it.  The one kernel that may start reading earlier (its inputs
are complete when it is allowed to start) does so past L1, which may hold lines of an earlier call."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_03961_b200", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s[^;{]*?(\w+)\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield os.path.basename(path), m.group(1), m.group(2), text[m.end():end - 1]


def test_kernels_are_found():
    names = [k[1] for k in _kernels()]
    assert {"plan_slots_kernel", "plan_summary_kernel", "gather_x_kernel", "router_dlogits_kernel", "split_w_kernel"} <= set(names)


@pytest.mark.parametrize("kernel", [k for k in _kernels() if "pdl_wait();" in k[3]], ids=lambda k: k[1])
def test_inputs_are_read_after_the_wait_or_past_l1(kernel):
    _, _, params, body = kernel
    inputs = re.findall(r"const\s[^,*]*\*\s*(?:__restrict__\s+)?(\w+)", params)
    early = re.sub(r"__ldcg\([^?:;]*", "", body[:body.index("pdl_wait();")])
    assert [n for n in inputs if re.search(rf"\b{n}\b(?!\s*[!=]=)", early)] == []
    if early != body[:body.index("pdl_wait();")]:              # __ldcg loses to a read-only load of the same pointer
        assert not re.search(r"const\s[^,*]*\*\s*__restrict__\s+(%s)\b" % "|".join(
            re.findall(r"__ldcg\((\w+)", body)), params)

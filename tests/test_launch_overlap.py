"""Source rules of the kernels that are resident while the launch in front of them still runs (they call
griddepcontrol.wait): what that launch writes must not be read through the read-only path, which is defined only for
data that does not change while the kernel lives and which a compiler may move across the wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_08065_b200", "csrc")
# its clearing kernel is an ordinary launch: everything it reads is complete before that one starts
BEHIND_AN_ORDINARY_LAUNCH = {"fused_stream_kernel"}


def strip_comments(src):
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", src, flags=re.S))


def closing(src, at, pair):
    depth = 0
    for i in range(at, len(src)):
        depth += (src[i] == pair[0]) - (src[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = strip_comments(open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?=const|uint16_t|double|int\b|float|void|Grad|Adam|Geometry)", src):
            end = closing(src, m.end() - 1, "()")
            if src[end + 1:].lstrip().startswith("{"):
                body = src.index("{", end)
                yield os.path.basename(path), m.group(1), src[m.end():end], src[body:closing(src, body, "{}") + 1]


def overlapping():
    found = [(f, n, p, b) for f, n, p, b in kernels() if "pdl_wait" in b or "griddepcontrol.wait" in b]
    return [k for k in found if k[1] not in BEHIND_AN_ORDINARY_LAUNCH]


def test_the_kernels_are_found():
    names = {n for _, n, _, _ in overlapping()}
    assert len(names) >= 25 and {"linear_tc_kernel", "plan_expand_kernel", "masked_adam_kernel", "compact_kernel"} <= names


@pytest.mark.parametrize("file,name,params,body", overlapping(), ids=lambda v: v if len(v) < 40 else "")
def test_no_read_only_loads(file, name, params, body):
    assert "__ldg(" not in body, f"{file}: {name}"
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params), f"{file}: {name}"


def test_tensor_memory_is_allocated_before_the_signal():
    """A dependent grid that is let in before a CTA has its tensor memory could take that memory and then wait for the CTA."""
    seen = set()
    for file, name, _, body in kernels():
        signal = re.search(r"pdl_launch_dependents|griddepcontrol\.launch_dependents", body)
        if "tcgen05.alloc" not in body or signal is None:
            continue
        # behind the meeting of the warps that follows the allocation, or behind the allocation in the allocating warp itself
        alloc = body.index("tcgen05.alloc")
        between = body[alloc:signal.start()]
        assert signal.start() > alloc and ("__syncthreads();" in between or "}" not in re.sub(r"\{[^{}]*\}", "", between)), f"{file}: {name}"
        seen.add(name)
    assert {"linear_tc_kernel", "gemm_pair_kernel", "gemm_split_kernel", "linear_gather_kernel", "gemm_tn_kernel",
            "linear_chain_kernel"} <= seen


def test_shared_helpers():
    src = strip_comments(open(os.path.join(CSRC, "bsp_common.cuh")).read())
    assert "__ldg(" not in src

"""`setmaxnreg` is defined only when all four warps of an aligned group execute the same instruction.  The kernels deal registers
by role, so the sources are read for every such instruction, the branches on the warp it stands in are evaluated for each warp,
and the warps that reach it have to be whole groups, each group reaching exactly one."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24011_b200", "csrc")
WARPS = 24


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _instructions(body):
    """Per setmaxnreg, the conditions on `warp` that lead to it: [(text, holds), ...]."""
    found, stack, closed = [], [], {}       # stack: conditions of the open blocks; closed: those of the last block of a depth
    for m in re.finditer(r"(else\s+)?if\s+(?:constexpr\s+)?\(((?:[^()]|\([^()]*\))*)\)\s*(\{)?|else\s*(\{)|(\{)|(\})|setmaxnreg", body):
        depth = len(stack)
        if m.group(0) == "setmaxnreg":
            found.append([c for block in stack for c in block])
        elif m.group(6):
            closed[depth - 1] = stack.pop()
        elif m.group(5):
            stack.append([])
        else:
            before = [(t, False) for t, _ in closed.get(depth, [])[-1:]] if m.group(1) or m.group(4) else []
            before = (closed.get(depth, [])[:-1] if before else []) + before
            if m.group(4):
                stack.append(before)
            elif m.group(3):
                stack.append(before + [(m.group(2), True)])
    return found


def _reached(conditions, names):
    def value(text, warp):
        text = re.sub(r"\b(?:RO|T)::", "", text)
        return eval(text, {"__builtins__": {}}, {**names, "warp": warp})     # comparisons of warp with a role's first warp
    about_warp = [(t, h) for t, h in conditions if re.match(r"\s*warp\b", t)]
    return [w for w in range(WARPS) if all(bool(value(t, w)) == h for t, h in about_warp)]


def _check(body, names):
    instructions = _instructions(body)
    assert len(instructions) == 3
    seen = []
    for c in instructions:
        warps = _reached(c, names)
        assert warps and len(warps) % 4 == 0 and all(w // 4 * 4 + i in warps for w in warps for i in range(4)), (c, warps)
        seen += warps
    assert sorted(seen) == list(range(WARPS))


def test_decode_kernel():
    s = _source("aq_decode_stack.cu")
    body = s[s.index("decode_stack_kernel(const DsArgs a) {"):s.index("struct DecodePlan")]
    unpack, collect = 8, 12
    names = {"DS_UNPACK_WARPS": unpack, "COLLECT0": unpack, "ISSUER": unpack + collect, "FEEDER": unpack + collect + 1,
             "RECORD0": unpack + collect + 2}
    _check(body, names)


def test_prefill_kernel():
    s = _source("aq_gemm.cu")
    body = s[s.index("gemm_kernel(const __grid_constant__"):s.index("tensor_map_encoder() {")]
    _check(body, {"GM_DQ_WARPS": 16, "GM_EP0": 16, "GM_TMA": 20, "GM_MMA": 21, "GM_PACKED": 22})


@pytest.mark.parametrize("split", (False, True))
def test_the_check_itself(split):
    branches = "if (warp < 8) { setmaxnreg } else if (warp == 20) { setmaxnreg } else if (warp >= 21) { setmaxnreg } else { setmaxnreg }"
    whole = "if (warp < 8) { setmaxnreg } else if (warp >= 20) { setmaxnreg if (warp == 20) { } else { } } else { setmaxnreg }"
    if split:
        with pytest.raises(AssertionError):
            _check(branches, {})
    else:
        _check(whole, {})

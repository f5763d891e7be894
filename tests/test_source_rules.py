"""Rules that the kernels' sources keep and that no run can show."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2011_05630_b200", "csrc")
CONSTANTS = {"w", "wp", "bias", "bias2", "b1", "bd", "b2"}   # weights, pointers into them, biases


def test_read_only_loads_are_for_weights_and_biases():
    """A kernel's CTAs start while the kernel before it still writes their input: what that one writes is not read through the
    read-only path, neither by __ldg nor through a const __restrict__ argument."""
    for name in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?\s*((?:\w+[.])*\w+)", src):
            assert m.group(1).split(".")[-1] in CONSTANTS, (name, m.group(0))
        for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", src):
            assert m.group(1) in CONSTANTS, (name, m.group(0))


def test_a_row_from_tensor_memory_is_waited_for_before_any_branch():
    """Until the wait a tensor-memory load's registers hold nothing; where the flow of control branches or goes back, the compiler may copy
    them.  The depthwise walk: every row that is asked for has landed before the next one, a way out of the loop or the loop's end."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "mbconv_lat.cu")).read())
    body = src[src.index("depthwise_task("):]
    body = body[:body.index("template <int STRIDE, bool RELU6, int SPLIT>")]
    assert not re.search(r"\bif\s*\([^;{]*\)\s*ld_row_issue", body)   # (in one branch alone: merged with the other's registers)
    walk = re.findall(r"\bnext\(\)|\bwait\(\)|\bbreak\b|\bwhile\b|\bfor\s*\(int j|\}", body[body.index("int rows = t.rows"):])
    for a, b in zip(walk, walk[1:]):
        assert (a == "next()") == (b == "wait()"), (a, b)
    assert walk.count("next()") == walk.count("wait()") >= 8

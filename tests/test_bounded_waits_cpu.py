"""Whoever leaves because a wait has run out leaves nobody behind at a barrier, which knows no limit: read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")


def _functions(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    for m in re.finditer(r"^(?:__device__|AS_DEV|__global__)[^;{}]*?\b(\w+)\([^;{}]*\)\s*\{", text, re.M):
        yield m.group(1), re.split(r"\n}\n", text[m.start():], maxsplit=1)[0]


def test_no_warp_returns_ahead_of_a_barrier_of_its_group():
    """A function of the query stage in which a warp may return by itself has no barrier of several warps behind that return, its own or one of a function that
    it calls."""
    functions = dict(_functions("tensor_qpass.cu"))
    assert {"q_softmax_unit", "q_leave_part", "q_merge_parts", "q_linear_unit"} <= set(functions)
    with_barrier = {name for name, body in functions.items() if "named_barrier_sync" in body}
    for name in ("q_softmax_unit", "q_leave_part", "q_merge_parts"):
        body = functions[name]
        returns = [m.start() for m in re.finditer(r"\breturn (?:false|make_float4\(0\.f, 0\.f, -1\.f)", body)]
        barriers = [m.start() for m in re.finditer(r"named_barrier_sync|" + "|".join(r"\b%s<" % f for f in with_barrier if f != name) or "$^", body)]
        assert not [b for b in barriers if (returns and min(returns) < b) or name != "q_softmax_unit"], name


def test_the_linear_unit_comes_to_all_its_barriers():
    """There the threads of a row's two halves meet: whoever's wait has run out goes on to the last barrier."""
    body = dict(_functions("tensor_qpass.cu"))["q_linear_unit"]
    assert body.rindex("named_barrier_sync") < body.index("return false") and body.count("return false") == 1

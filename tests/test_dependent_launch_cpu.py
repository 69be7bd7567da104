"""What kernels that set up beside the kernel before them may touch ahead of their wait for it, read from the sources: a run shows a fault only where that
kernel lets dependents in before it writes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")
# the handle's own memory: a table that does not change, and the status word
OWN = {"sm_rank", "status"}
# reached by warps only that have waited where the rest have not yet (the key stage's gather warps)
BEHIND_A_WAIT_OF_THEIR_WARPS = {"kpass_kernel": {"ks_w", "vs_w"}}


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                yield re.sub(r"//[^\n]*", "", f.read())


def _pointers():
    """Names of the pointer members of the kernels' parameters."""
    found = set()
    for text in _sources():
        for members in re.findall(r"\bstruct \w+ \{(.*?)\n?\};", text, re.S):
            found |= set(re.findall(r"\*\s*(\w+)\s*[,;]", members))
    return found


def _kernels():
    """(name, text from the name to the closing brace) of the kernels with a wait for the kernel before them, comments removed."""
    found = []
    for text in _sources():
        for body in re.split(r"\b__global__\b", text)[1:]:
            body = re.sub(r"^.*?(\w+)\((?=const|[A-Z])", r"\1(", re.sub(r"__launch_bounds__\([^\n]*?\)+\s", "", re.split(r"\n}\n", body, maxsplit=1)[0]), count=1, flags=re.S)
            if "griddep_wait()" in body:
                found.append((body[:body.index("(")], body))
    return found


def _without_helpers(text):
    """The text with each local function that it defines put in where it is called."""
    while True:
        m = re.search(r"auto (\w+) = \[&\]\([^)]*\)[^{;]*\{", text)
        if m is None:
            return text
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        rest = text[at:]
        text = text[:m.start()] + re.sub(r"\b%s\(" % m.group(1), lambda _: "{" + text[m.end():at - 1] + "} (", rest)


def _early(name, body):
    """Pointers of the parameters that are used, but to ask whether they are there, ahead of the last wait."""
    body = _without_helpers(body)
    ahead = body[:body.rindex("griddep_wait()")]
    used = set(re.findall(r"\bp\.(\w+)\b(?!\s*[!=]= nullptr)", ahead)) & _pointers()
    return used - OWN - BEHIND_A_WAIT_OF_THEIR_WARPS.get(name, set())


def test_nothing_of_the_callers_is_touched_ahead_of_the_wait():
    kernels = _kernels()
    assert len(kernels) >= 10 and "kpass_kernel" in dict(kernels) and {"bias", "ks_w", "z", "part_dS"} <= _pointers()
    assert {name: _early(name, body) for name, body in kernels if _early(name, body)} == {}


def test_the_rule_sees_an_early_load():
    """Of a bias, straight or through a local function."""
    assert _early("k", "k(const P p) {\n const float b = p.bias[0];\n griddep_wait();") == {"bias"}
    assert _early("k", "k(const P p) {\n auto get = [&](int i) { return p.bias[i]; };\n get(1);\n griddep_wait();") == {"bias"}
    assert _early("k", "k(const P p) {\n auto get = [&](int i) { return p.bias[i]; };\n griddep_wait();\n get(1);") == set()

"""What kernels that set up beside the kernel before them may touch ahead of their wait for it, read from the sources: a run shows a fault only where that
kernel lets dependents in before it writes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")
# the handle's own memory: a table that does not change, the status word, and a counter that only CTAs use that have not yet let dependents in
OWN = {"sm_rank", "status", "part_ticket"}
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


# kernels that look at the status word, and what has to stand between their second look and all that they write
SECOND_LOOK = {
    "kpass_kernel": r"late = gathers \|\| warp == 11 \? status_now\(p\.status\)[^}]*", "phi1_kernel": r"bool live = __all_sync\(0xffffffffu, status_clear\(",
    "phi1_run_kernel": r"bool ok = __all_sync\(0xffffffffu, status_clear\(", "qlin_kernel": r"start && u < n_grp; \+\+u\)\s*if \(!q_linear_unit<",
    "qpass_kernel": r"start && u < n_grp; \+\+u\)\s*if \(!q_softmax_unit<", "qstream_kernel": r"if \(__all_sync\(0xffffffffu, status_clear\([^;]*\)\) qs_compute\(",
    "btq_kernel": r"late = status_now\(p\.status\)", "btk_kernel": r"late = status_now\(p\.status\)", "bsq_kernel": r"late = status_now\(p\.status\)",
    "bsk_kernel": r"late = status_now\(p\.status\)"}
WRITES = r"tma_store_3d\(|\bout\[\(size_t\)r \* LPR|p\.part_z\[|\(to \+ \(size_t\)rank|\\batomicAdd\(cnt|bt_store_acc\(\w|p\.part_\w+\[slot|" \
         r"reinterpret_cast<float4\*>\(dst\)\[|\bdst\[i\] =|copy_rows<D>\(|q_softmax_unit<|q_linear_unit<|qs_compute\("


def test_a_time_out_of_the_kernel_before_is_seen_ahead_of_the_first_write():
    """The status word is looked at again behind the wait (the look beside the kernel before it may come too early), by all that write and before they do."""
    kernels = dict(_kernels())
    assert {name for name, body in kernels.items() if "s_skip" in body or "*skip" in body} == set(SECOND_LOOK)
    for name, look in sorted(SECOND_LOOK.items()):
        body = kernels[name]
        body = body[body.index("if (warp >= 8) griddep_wait();") if name == "kpass_kernel" else body.rindex("griddep_wait()"):]
        at = re.search(look, body)
        writes = [m.start() for m in re.finditer(WRITES, body)]
        assert at and writes and at.start() < min(writes), (name, at, writes[:3])
        for x in writes:
            assert "s_late != 0u) return" in body[:x] or re.search(r"late == 0u|late != 0u \? -1|live && |\bif \(ok(?: && |\) copy_rows)|while \(ok && |start &&|status_clear\(", body[:x][-1300:]), (
                name, body[:x][-300:])
        assert ("status_again(" in body) == ("status_clear(" in body), name

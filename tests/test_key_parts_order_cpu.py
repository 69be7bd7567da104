"""Which CTA a CTA of the query stage's last round is, where key loops go in parts: CUDA promises no order in which CTAs start, and one that waits for another's part
must not wait for one that cannot start before it has ended."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")


def test_parts_go_by_the_order_in_which_ctas_have_started():
    with open(os.path.join(CSRC, "tensor_qpass.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    for name in ("q_leave_part", "q_merge_parts", "q_parts"):
        body = re.split(r"\n}\n", text[re.search(r"\b%s\(const QParams& p[^;{]*\{" % name, text).start():], maxsplit=1)[0]
        assert "blockIdx" not in body, name
    # taken ahead of what lets the next launch's CTAs start: these take theirs from the same counter
    kernel = text[text.index("\nqpass_kernel("):]
    assert kernel.index("atomicInc(p.part_ticket, gridDim.x - 1u)") < kernel.index("griddep_launch();") < kernel.index("griddep_wait();")

"""The batched sort of ensemble members changes a member's work-unit size only
together with its unit list: a size that does not belong to the list sends the
tile kernel past the ends of its bins.  An allocation that fails between the
two is not something a test can bring about on a GPU, so the order is checked
in the source."""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1407_1810_gb300", "csrc", "particles32.cu")


def test_unit_size_is_set_after_the_last_call_that_can_fail():
    s = open(SRC).read()
    body = s[s.index("int ens_sort32("):]
    body = body[: body.index("\n}\n")]
    last = max(m.end() for m in re.finditer(r"PIC_CUDA\(", body))
    for state in (r"T\.unit\s*=", r"mix_sort\s*=", r"std::swap\(c->p32", r"n_used\s*=[^=]"):
        at = [m.start() for m in re.finditer(state, body)]
        assert at and min(at) > last, state

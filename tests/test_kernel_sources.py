"""What the sources of the kernels must hold to and no run can show."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_12260_b200", "csrc")


def _calls(text, name):
    """The argument texts of every call of `name`."""
    for m in re.finditer(r"\b%s\(" % re.escape(name), text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def test_a_round_does_not_read_its_tables_through_the_read_only_path():
    """The search's first kernel starts beside the kernel that writes the speedup tables, so the tables are
    not read-only for its lifetime, which is what __ldg (ld.global.nc) asks for, wait or no wait."""
    text = open(os.path.join(CSRC, "round_flow.cu")).read()
    assert "griddepcontrol.wait" in text
    args = list(_calls(text, "__ldg"))
    assert args                                             # (the scan finds calls at all)
    assert [a for a in args if "table" in a] == []
    assert any("table" in a for a in _calls(text, "__ldcg"))

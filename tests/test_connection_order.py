"""The connection drops the edges of undecided cells by moving the others up
in place: every lane reads its edge before any lane writes (CPU: the source;
a ballot orders the lanes, not their shared memory)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_edges_are_read_by_all_lanes_before_any_moves_up():
    src = open(os.path.join(ROOT, "paper_2008_13461_gb300", "csrc", "pt_connect.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    body = code[code.index("int write_edges("):code.index("int test_candidates(")]
    moves = [m.start() for m in re.finditer(r"sm\.acc_pos\[[^\]]*\]*\] = ", body)]
    assert len(moves) == 2
    for at in moves:
        read = max(m.start() for m in re.finditer(r"= i < \w+ \? sm\.acc_pos\[", body[:at]))
        assert "__syncwarp();" in body[read:at]

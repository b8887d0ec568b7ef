"""The polling phase's lanes hand values to one another inside one launch: every
access to a word that another lane writes has to be a strong one (relaxed, at
device scope), in the source's terms one of the poll_* accessors."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_12800_gb300", "csrc")


def _polling():
    s = open(os.path.join(CSRC, "fr_engine.cuh")).read()
    begin = s.index("constexpr int kPollCells")
    return s[begin:s.index("// Blocks of a cooperative launch", begin)]


def test_polling_accesses_are_strong():
    s = _polling()
    # the accessors: relaxed at device scope, nothing else touches the arrays
    for op in ("ld.relaxed.gpu.global.f32", "st.relaxed.gpu.global.f32", "ld.relaxed.gpu.global.u64",
               "st.relaxed.gpu.global.u64"):
        assert s.count(op) == 1
    begin = s.index("ready = true")
    steps = s[begin:]
    weak = re.findall(r"\b(?:wr_f|wr_area|rd_cg|rd_area|ld_cg|__ldcg\(P|g_value<E>|P\.(?:out_hi|out_lo|area)\b)", steps)
    assert not weak, weak
    assert all(f in steps for f in ("poll_value(", "poll_put(", "poll_area(", "poll_put_area("))

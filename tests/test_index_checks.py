"""The index-checking build covers the pair kernel: in process_tile_sym every access
to a shared or a global array goes by RT_IDX or RT_AT, or by an index that came
out of one (the cell c, a staged cell cc, a place in the box at)."""
import os
import re

HERE = os.path.dirname(os.path.abspath(__file__))
KERNEL = os.path.join(os.path.dirname(HERE), "paper_1403_6126_gb300", "csrc", "rt_step_sym.cuh")
ARRAYS = r"s_\w+|c_al|c_v|l_al|l_v|F|Fl|fc|In|IV|out|a\.(?:ang|inflow|I_in|I_out|cen_in|mom_in|sa|ss|v)|a\.alpha\[\d\]|\w+\(I\)|\(s_tab\)"
CHECKED = r"(?:d \* N \+ )?(?:cc|c)|at"
POINTERS = r"s_I|s_F|s_IV|s_fc|s_tab|In|IV|F|Fl|fc|out"


def _body():
    text = open(KERNEL).read()
    start = text.index("process_tile_sym(const StepArgs")
    end = text.index("\n}\n", start)
    return re.sub(r"//[^\n]*", "", text[start:end])


def test_every_access_of_the_pair_kernel_is_checked():
    body = _body()
    subscripts = re.findall(r"(?<![\w.>])(%s)\[(.*)" % ARRAYS, body)
    assert len(subscripts) > 25
    loose = [(a, s) for a, s in subscripts
             if not s.startswith("RT_IDX(") and not re.match(r"(?:%s)\]" % CHECKED, s)]
    assert not loose, loose
    # arrays reached through a pointer that walks
    for walk in (r"x = RT_AT\(x, In", r"v = RT_AT\(v, IV", r"\*RT_AT\(fc \+", r"\*RT_AT\(Fl \+", r"RT_AT\(from\("):
        assert re.search(walk, body), walk
    assert not re.search(r"\*\((?:%s) \+" % POINTERS, body)

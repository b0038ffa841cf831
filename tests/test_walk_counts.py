"""The walk counts interpreted nodes and levels for statistics that are 64 bits
wide.  A warp's own counts are 32 bits wide, so they are emptied into the totals
between two children.  (More than 2^32 nodes by one warp in one generation
cannot be had in a test: the source is read.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_counts_are_wide_or_emptied_between_children():
    src = open(os.path.join(ROOT, "paper_2205_03251_gb300", "csrc", "generation.cuh")).read()
    code = re.sub(r"//[^\n]*", "", src)
    body = code[code.index("k_walk(DevPop d"):code.index("struct OnePassEvalLayout")]
    m = re.search(r"(uint32_t|unsigned long long) (st_interp = 0[^;]*);", body)
    names = re.findall(r"st_\w+", m.group(2))
    assert len(names) == 4
    if m.group(1) == "uint32_t":
        child = body.index("for (;;) {", m.end())
        take = body.index("atomicAdd(&d.q[wr.qctr]", child)
        head = body[child:take]
        assert re.search(r"if \(\(" + r" \| ".join(names) + r"\) >> 31\) tally\(\);", head)
        empty = body[body.index("auto tally"):child]
        for n in names:
            assert re.search(r"atomicAdd\(&g\.gstat\[\w+\], \(unsigned long long\)" + n + r"\)", empty), n
        assert " = ".join(names) + " = 0;" in empty

"""An incremental walk ends at the child's root, stopped, or with an error: when
the cached links of the mother lead past the root, the value at hand is an inner
subtree's and must not become the child's fitness.  No call of the library can
make such links, so the walk's ways out are read in the source."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_way_out_of_the_combination():
    src = open(os.path.join(ROOT, "paper_2205_03251_gb300", "csrc", "generation.cuh")).read()
    code = re.sub(r"//[^\n]*", "", src)
    start = code.index("while (!fail) {", code.index("k_walk(DevPop d"))
    depth, end = 0, start
    for end in range(code.index("{", start), len(code)):
        depth += {"{": 1, "}": -1}.get(code[end], 0)
        if depth == 0:
            break
    body = code[start:end]
    exits = [m.start() for m in re.finditer(r"\bbreak;", body)]
    assert len(exits) >= 3
    for at in exits:
        before = " ".join(body[:at].split())
        assert (before.endswith("if (fail)") or                        # an earlier failure
                before.endswith("if (D.p == 0)") or                    # the root is combined
                re.search(r"if \(stopped_w && \([^;{]*\)$", before) or    # stopped: nothing above needs a value
                before.endswith("fail = true;") or                     # an error
                re.search(r"if \(!stopped_w && c != 0\) \{.{0,120}fail = true; \}$", before)), before[-200:]

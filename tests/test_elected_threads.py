"""Which lane `elect.sync` elects is not specified.  A region for one elected thread may therefore not have an alternative that is entered
by lane number: if that lane is the elected one, nobody runs the alternative and every wait on it runs out."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_12128_b200", "csrc")


def block_end(text, start):
    depth = 0
    for i in range(text.index("{", start), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return i + 1


def test_no_lane_number_beside_an_elected_thread():
    regions = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        elected = {"elect_one()"} | {m.group(1) for m in re.finditer(r"\bbool (\w+) = elect_one\(", text)}
        for name in elected:
            for m in re.finditer(r"\bif \([^;{]*?" + (re.escape(name) if "(" in name else rf"\b{name}\b") + r"[^;{]*\{", text):
                regions += 1
                rest = text[block_end(text, m.start()):]
                alternative = re.match(r"\s*else\s*if\s*\(([^{]*)\{", rest)
                assert not (alternative and re.search(r"\blane\s*[=!<>]=?\s*\d", alternative.group(1))), (os.path.basename(path), m.group(0))
                assert alternative or not re.match(r"\s*else\b", rest), (os.path.basename(path), m.group(0))
    assert regions > 30

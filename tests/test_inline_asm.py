"""Inline assembly that touches memory or orders it is volatile and names memory
as clobbered: without both the compiler may move it across stores, barriers
and griddepcontrol.wait (a load that is neither reads words of another phase)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1101_1427_gb300", "csrc")
MEMORY = re.compile(r"(?:^|[\s{;\"])(ld|st|red|atom|griddepcontrol\.wait|fence|membar|cp|mbarrier|barrier)\b[.;]?")


def statements():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\basm\b\s*(volatile)?\s*\(", text):
            depth, k = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[k], 0)
                k += 1
            yield os.path.basename(path), bool(m.group(1)), text[m.end():k - 1]


def test_memory_assembly_is_ordered():
    seen = 0
    for name, volatile, body in statements():
        if MEMORY.search(re.split(r'"\s*:', body)[0] + '"'):
            seen += 1
            assert volatile and '"memory"' in body, (name, body)
    assert seen >= 5

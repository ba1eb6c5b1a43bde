"""Rules of the kernel sources that only reading shows broken."""
import glob
import os
import re

import paper_2510_06873_gb300 as pkg

CSRC = os.path.join(os.path.dirname(pkg.__file__), "csrc")


def test_assembly_that_touches_memory_is_ordered():
    """A load that the compiler takes for a function of its address may move
    before griddepcontrol.wait or a fence, where an earlier kernel or another
    block is still writing.  Assembly that loads, stores or waits is therefore
    volatile with a memory clobber, and the toolkit's cache-hint loads, which
    promise neither, are not used."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        assert not re.search(r"__ld(cs|cg|ca|lu|cv)\s*\(", text), path
        for m in re.finditer(r"\basm\b(\s+volatile)?\s*\((.*?)\)\s*;", text, flags=re.S):
            if re.search(r"\"\s*(ld|st|atom|red|cp|griddepcontrol|membar|fence)\b", m.group(2)):
                seen += 1
                assert m.group(1) and '"memory"' in m.group(2), (path, m.group(0))
    assert seen >= 3

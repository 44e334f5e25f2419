"""Inline assembly that reads or writes memory through an address operand says so
to the compiler: without a "memory" clobber its order against ordinary loads and
stores of the same locations is not fixed."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_assembly_that_touches_memory_has_a_memory_clobber():
    seen = 0
    for path in glob.glob(os.path.join(ROOT, "paper_2408_14558_gb300", "csrc", "*.cu*")):
        for stmt in re.findall(r'\basm\b\s*(?:volatile\s*)?\((.*?)\)\s*;', open(path).read(), re.S):
            if re.search(r'"\s*[^"]*\b(?:ld|st|atom|red|cp)\.[^"]*\[', stmt):
                seen += 1
                assert '"memory"' in stmt, f"{os.path.basename(path)}: {stmt}"
    assert seen >= 4

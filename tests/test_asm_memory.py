"""Inline PTX that reads or writes memory, or orders accesses to it, says so to the
compiler, which else may move or drop the plain accesses around it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), '..', 'paper_2003_01490_gb300', 'csrc')
TOUCHES = re.compile(r'(?<![\w.])(ld|st|atom|red|cp|ldmatrix|stmatrix|mbarrier|barrier|fence|membar)\.')


def statements(text):
    """The argument lists of the file's asm statements."""
    for m in re.finditer(r'\basm\s*(volatile)?\s*\(', text):
        depth, k = 1, m.end()
        while depth:
            depth += {'(': 1, ')': -1}.get(text[k], 0)
            k += 1
        yield text[m.end():k - 1]


def test_asm_statements_that_touch_memory_declare_it():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, '*.cu')) + glob.glob(os.path.join(CSRC, '*.cuh'))):
        with open(path) as f:
            for s in statements(f.read()):
                if TOUCHES.search(s.replace('\\n', ' ').replace('\\t', ' ')):
                    found += 1
                    assert '"memory"' in s, (os.path.basename(path), s)
    assert found >= 3

"""Inline assembly that touches memory says so: without the "memory" clobber the compiler may move other accesses across the
statement - a read of shared memory ahead of the wait that it depends on, for instance."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_05534_b200", "csrc")
# loads, stores, atomics, bulk copies, barriers, fences and the tensor core's instructions (a prefetch changes nothing)
TOUCHES = re.compile(r'"[^"]*?\b(ld|st|red|atom|cp|mbarrier|barrier|bar|fence|griddepcontrol|tcgen05|multimem)\.[a-z]')


def _asm_statements(text):
    for m in re.finditer(r"\basm\s*(volatile)?\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text.count("\n", 0, m.start()) + 1, text[m.start():i]


def test_every_statement_that_touches_memory_names_it():
    seen, bad = 0, []
    for name in sorted(os.listdir(CSRC)):
        for line, stmt in _asm_statements(open(os.path.join(CSRC, name)).read()):
            # (the two statements assembled from macros spell their loads in the macros; their own text has tensor-memory reads)
            if not TOUCHES.search(stmt):
                continue
            seen += 1
            if '"memory"' not in stmt or "volatile" not in stmt:
                bad.append("%s:%d" % (name, line))
    assert seen > 30 and not bad, (seen, bad)

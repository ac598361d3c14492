"""Rules of the device code that no run can show to be kept: what a broken one does depends on the compiler or on a wait that
runs out at the wrong moment."""
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
    """Without the "memory" clobber the compiler may move other accesses across the statement: a read of shared memory ahead of
    the wait that it depends on, for instance."""
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


def test_waits_before_warp_wide_operations_are_the_whole_warps():
    """A wait of each lane for itself may end differently for the lanes of a warp when it runs out; votes, shuffles and
    tensor-memory reads would then wait for lanes that have left.  Such waits are for threads that do none of these (the weight
    builders of the tensor-core merge, the self-test) or whose way does not depend on what the wait returns until they have voted
    (the second scoring pass)."""
    per_lane = {}
    for name in sorted(os.listdir(CSRC)):
        n = len(re.findall(r"(?<!bool )\bmbar_wait\(", open(os.path.join(CSRC, name)).read()))
        if n:
            per_lane[name] = n
    assert per_lane == {"flowmm_api.cu": 1, "merge_tc.cuh": 2, "tc_stream.cuh": 2}, per_lane
    assert {name for name in os.listdir(CSRC) if "S::quad_extra_wait_lanes(" in open(os.path.join(CSRC, name)).read()} == {"score_tc.cuh"}


def test_no_block_leaves_or_reports_before_its_predecessor_is_done():
    """Kernels are launched as programmatic dependents: a block that returned without waiting would let the kernel after it start
    before the kernel in front has ended, and a status word may still be the predecessor's."""
    bad = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__global__[^;{]*\{", text):
            body = text[m.end():]
            body = body[:re.search(r"\n}", body).start()]
            wait = min((body.find(w) for w in ("predecessor_done()", "::setup(") if w in body), default=-1)
            early = re.search(r"\breturn\b|atomicCAS|status_write|atomicAdd", re.sub(r"\[&\][^{]*\{[^}]*\}", lambda l: " " * len(l.group()), body))
            if wait < 0 or (early and early.start() < wait):
                bad.append("%s:%d" % (name, text.count("\n", 0, m.start()) + 1))
    assert not bad, bad

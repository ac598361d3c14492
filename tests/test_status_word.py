"""The status word of a decode call: every block of the call may report before, after or without the block that clears it, on
a workspace with any content.  The transitions are plain functions, compiled here for the host and run in every order."""
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <stdio.h>
#include "status_word.cuh"
int main() {
    unsigned long long word;
    unsigned call;
    int n, code;
    while (scanf("%llx %x %d", &word, &call, &n) == 3) {
        for (; n > 0; --n) {
            if (scanf("%d", &code) != 1) return 1;
            word = code == 0 ? flowmm::status_cleared(word, call) : flowmm::status_reported(word, call, code);
        }
        printf("%llx\n", word);
    }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("status")
    (d / "s.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_05534_b200", "csrc"), "-o", str(d / "s"), str(d / "s.cpp")])

    def go(cases):
        text = "".join("%x %x %d %s\n" % (w, c, len(e), " ".join(map(str, e))) for w, c, e in cases)
        return [int(x, 16) for x in subprocess.run([str(d / "s")], input=text, capture_output=True, text=True, check=True).stdout.split()]
    return go


def test_no_order_of_clearing_and_reporting_loses_a_report(run):
    call, other = 0x9E3779B1, 0x3C6EF362
    before = [0, 0x4D4D4D4D4D4D4D4D, other << 32, (other << 32) | 8, (1 << 64) - 1, 8]    # fresh, garbage, an earlier call's, its error
    cases = [(w, call, e) for w in before for events in ([0], [0, 8], [0, 8, 6]) for e in itertools.permutations(events)]
    for (word, _, events), after in zip(cases, run(cases)):
        reports = [e for e in events if e]
        assert after & 0xFFFFFFFF == (reports[0] if reports else 0), (hex(word), events, hex(after))
        assert after >> 32 == call

"""A kernel that is resident while the one before it still writes the state
reads that state with plain loads.  __ldg (Store<>::ld, PairIO<>::ld) promises
that nobody writes the data during the kernel's lifetime, so the compiler may
move it above the wait; constant tables may keep it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_03271_gb300", "csrc")
WAIT = re.compile(r"(?<!void )\b(?:chain_wait|dependency_wait)\([^)\n]*\);")
STATE = re.compile(r"\b(?:Store|PairIO|RawPair)<\w+>::(?:ld|two)\(|__ldg\((?!\w+ \+|reinterpret_cast<const float4\*>\(A\.rowtab)")


def test_state_loads_of_chained_kernels_are_plain():
    checked = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in WAIT.finditer(text):
            body = text[m.end():text.index("\n}\n", m.end())]
            if body.lstrip().startswith("return;"):  # a CTA with nothing to do
                continue
            hit = STATE.search(body)
            assert hit is None, (os.path.basename(path), hit and body[hit.start():hit.start() + 60])
            checked += 1
    assert checked == 5  # the paired tile; start, both one-cell kernels and the one-population kernel of the two launches

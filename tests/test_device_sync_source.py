"""The inline-PTX synchronisation helpers keep the compiler from moving memory accesses
across them: without a "memory" clobber a plain store may rise above the wait that says
its buffer is free."""
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1605_01020_gb300", "csrc")
ORDERING = ("mbarrier.", "fence.", "tcgen05.fence", "tcgen05.commit", "tcgen05.wait", "cp.async.bulk", "bar.sync", "bar.arrive",
            "barrier.", "ld.acquire")


def test_ordering_instructions_clobber_memory():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"asm volatile\s*\((.*?)\);", text, re.S):
            if any(op in m.group(1) for op in ORDERING):
                seen += 1
                assert '"memory"' in m.group(1), f"{name}: {m.group(1)[:80]}"
    assert seen > 10

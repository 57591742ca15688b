"""A wait that gives up must not let its CTA return while a bulk copy is still
on its way into the CTA's shared memory: every barrier a bulk copy completes is
waited for with cta_wait, which repeats a wait that gave up before it reports
it.  A copy that never arrives cannot be staged without a GPU fault, so the
sources are read instead."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_05552_gb300", "csrc")


def test_bulk_copies_are_waited_for_twice():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for bar in set(re.findall(r"bulk_load\([^;]*?(&S\.\w+)\);", text)):
            found += 1
            assert re.search(r"\bcta_wait\(" + re.escape(bar) + r"\b", text), (name, bar)
            assert not re.search(r"\bmbar_wait\(" + re.escape(bar) + r"\b", text), (name, bar)
    assert found
    body = re.search(r"bool cta_wait\(.*?\n}\n", open(os.path.join(CSRC, "pdn_surrogate.cu")).read(), re.S).group(0)
    assert len(re.findall(r"mbar_wait\(bar, phase, kMaxPolls\)", body)) == 2 and "return false" in body

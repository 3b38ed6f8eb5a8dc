"""The checked build's claim that the kernels' global stores test their index, as far as the sources show it: every store site is
used, and the trace, which several roll-out kernels write, is written by the two checked functions only."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_05008_b200", "csrc")


def _sources():
    return {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.[ch]*"))}


def test_every_store_site_is_checked_somewhere():
    text = _sources()
    sites = re.findall(r"(EVO_SITE_\w+) = \d+", text["internal.h"])
    assert len(sites) >= 8
    everything = "".join(text.values())
    for site in sites:
        assert re.search(r"EVO_IN_BOUNDS\([^;]*\b%s\b" % site, everything), site


def test_the_trace_is_written_by_checked_stores_only():
    stores = [(name, line.strip()) for name, body in _sources().items() for line in body.splitlines()
              if re.search(r"\ba\.trace(\[| \+ )", line)]
    assert stores and {name for name, _ in stores} == {"tasks.cuh"}, stores
    assert all(re.search(r"a\.trace(\[at\]| \+ at\))", line) for _, line in stores)

"""A bounded wait that expired is reported as RABITQ_ETIMEOUT wherever it was, and
the bucket-major scan's under its own name. Read from the source: no input makes
a wait expire."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2405_12497_gb300", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, f.read()


def test_expired_waits_are_timeouts():
    seen = 0
    for name, text in _sources():
        for m in re.finditer(r'fail\(\s*(RABITQ_\w+),\s*"([^"]*expired[^"]*)"', text):
            assert m.group(1) == "RABITQ_ETIMEOUT", (name, m.group(0))
            seen += 1
    assert seen >= 6


def test_the_scan_reports_its_own_waits():
    text = dict(_sources())["kernels_bucket.cu"]
    flags = re.findall(r"atomicExch\(P\.err, (\w+)\)", text)
    assert flags == ["kErrScanWait"]

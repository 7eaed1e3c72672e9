"""Each translation unit has its own device error flag: the check must read every one that a wait can raise."""

import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2607_12358_gb300" / "csrc"


def test_every_unit_that_waits_is_read():
    check = (CSRC / "capi.cu").read_text()
    check = check[check.index("acid_status acid_check_device_error"):]
    check = check[:check.index("\n}")]
    waiting = [p for p in sorted(CSRC.glob("*.cu")) if re.search(r"\bmbar_wait|g_device_error", p.read_text())]
    assert len(waiting) >= 3
    for path in waiting:
        reader = re.search(r"^ACID_DEVICE_FLAG_READER\((\w+)\)", path.read_text(), re.M)
        assert reader, path.name
        assert reader.group(1) + "()" in check, path.name

"""Launch shapes follow the device's SM count: no source takes it for granted."""
import glob
import os
import re

from paper_2211_14318_gb300 import build as b


def test_no_literal_sm_count():
    for path in sorted(glob.glob(os.path.join(b.CSRC, "*.cu*")) + glob.glob(os.path.join(b.CSRC, "*.h"))):
        for k, line in enumerate(open(path), 1):
            assert not re.search(r"\b(152|148|132)\b", line.split("//")[0]), f"{os.path.basename(path)}:{k}"

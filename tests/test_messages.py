"""What the library says of itself names nothing that is not there any more."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GONE = re.compile(r"\bTMA\b|staged kernel|autotun|tile list|shared-memory path|bulk kernel|geq_pairs", re.I)


def test_sources_and_header_name_no_removed_kernel():
    csrc = os.path.join(ROOT, "paper_1410_3464_gb300", "csrc")
    files = [os.path.join(csrc, f) for f in sorted(os.listdir(csrc)) if f.endswith((".cu", ".cuh", ".h"))]
    for path in files + [os.path.join(ROOT, "include", "pslbm.h"), os.path.join(ROOT, "paper_1410_3464_gb300", "pslbm.py")]:
        with open(path) as f:
            for n, line in enumerate(f, 1):
                assert not GONE.search(line), f"{os.path.basename(path)}:{n}: {line.strip()}"

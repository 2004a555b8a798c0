"""A context works on one stream, which may be a non-blocking one: copies and fills of the device data that
its kernels read go through that stream, not through the legacy stream (nothing orders the two)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_09782_gb300", "csrc")


def test_no_copy_or_fill_on_the_legacy_stream():
    """vgtb_diag.cu alone launches on the legacy stream, and copies there too."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        if os.path.basename(path) == "vgtb_diag.cu":
            continue
        with open(path) as f:
            for no, line in enumerate(f, 1):
                if re.search(r"\bcuda(Memcpy|Memset|MemcpyToSymbol|Memcpy2D|Memset2D)\(", line.split("//")[0]):
                    found.append(f"{os.path.basename(path)}:{no}")
    assert not found, found

"""The bench's roofline names the distance kernel that the profiled fits ran (CPU)."""
import glob
import hashlib
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


class Prof:
    def __init__(self, launches, n, d, k, ms):
        self.assign_launches = launches
        self.assign_ms = ms
        self.assign_flops = 2.0 * n * k * d * launches
        self.assign_bytes = 4.0 * n * d * launches


def _roof(d, k, screened, launches=10):
    return bench.roofline_of("fp32", d, k, Prof(launches, 1_000_000, d, k, 5.0), None, None, screened)


def test_kernel_is_the_one_that_ran():
    # the centers of these shapes do not fit beside the screen's rings, or most rows
    # stayed open: no launch, or a stage's first one only, went through it
    assert _roof(128, 448, 0)["kernel"] == "assign_large"
    assert _roof(8, 32, 0)["kernel"] == "assign_small<8>"
    assert _roof(8, 32, 1)["kernel"] == "assign_small<8>"
    for d, k in ((128, 448), (8, 32)):
        assert _roof(d, k, 0)["bound"] == "alu"


def test_screened_fits():
    r = _roof(8, 32, 10)
    assert r["kernel"] == "assign_mma_ring<8>" and r["bound"] == "hbm" and r["unit"] == "GB/s"
    assert abs(r["achieved"] - 10 * 32e6 / 5e-3 / 1e9) < 1e-6 * r["achieved"]
    assert _roof(12, 16, 9)["kernel"] == "assign_mma_ring<16>"
    assert _roof(100, 60, 10)["kernel"] == "assign_mma_ring<128>"
    assert _roof(16, 1000, 10)["bound"] == "tensor"


def test_dram_lines_of_the_screen_match_its_source():
    """'dram-per-point: <kernel> <bytes> <sha256>' lines, like the traffic-per-point
    lines of the other kernels, count only for the source they were captured on."""
    src = os.path.join(ROOT, "paper_1108_1351_gb300", "csrc", "assign_mma.cu")
    with open(src, "rb") as fh:
        sha = hashlib.sha256(fh.read()).hexdigest()
    for md in glob.glob(os.path.join(ROOT, "profiles", "*.md")):
        with open(md) as fh:
            for line in fh:
                parts = line.strip().strip("`").split()
                if len(parts) == 4 and parts[0] == "dram-per-point:":
                    assert parts[1].startswith("assign_mma_ring<") and parts[3] == sha, md
                    assert float(parts[2]) > 0

"""bench.py's DRAM traffic: scaled from an ncu capture of the kernels as they
stand, and not given for kernels that have changed since."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

LEDGER = {"n_cross": 3_000_000, "n_peel_cross": 2_000_000}


def test_traffic_of_the_captured_kernels(monkeypatch):
    monkeypatch.setattr(bench, "NCU_KERNEL_DIGEST", bench.kernel_digest())
    t, p = bench.captured_traffic(LEDGER)
    assert t == pytest.approx(3e6 * bench.NCU_TRACE_BYTES_PER_CROSSING)
    assert p == pytest.approx(2e6 * bench.NCU_PEEL_BYTES_PER_CROSSING)


def test_no_traffic_of_other_kernels(monkeypatch, tmp_path):
    """A changed statement in any of the captured sources leaves the figure
    out; comments and white space do not."""
    csrc = tmp_path / "paper_1206_3710_gb300" / "csrc"
    csrc.mkdir(parents=True)
    src = os.path.join(ROOT, "paper_1206_3710_gb300", "csrc")
    for n in os.listdir(src):
        (csrc / n).write_bytes(open(os.path.join(src, n), "rb").read())
    monkeypatch.setattr(bench, "NCU_KERNEL_DIGEST", bench.kernel_digest())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    f = csrc / "rt_device.cuh"
    text = f.read_text()
    f.write_text(text + "\n// a remark\n/* and\nanother */\n")
    assert bench.captured_traffic(LEDGER) != (None, None)
    f.write_text(text + "\nstatic int one;\n")
    assert bench.captured_traffic(LEDGER) == (None, None)


def test_line_asks_for_the_capture():
    """The line's traffic comes from captured_traffic alone."""
    text = open(os.path.join(ROOT, "bench.py")).read()
    body = text[text.index("def parse("):]
    assert "captured_traffic(" in body and "NCU_" not in body

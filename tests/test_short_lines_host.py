"""The two-stage plans of 32, 48 and 80 points on the CPU: each twiddle as near to its root as a table entry is, and the
transforms against an FP64 DFT."""
from test_layout_host import build_and_run


def test_short_lines(tmp_path):
    out = build_and_run("host_short_lines_check.cu", tmp_path / "short_lines")
    assert out.count("rms rel error") == 3 * 3 and out.count("twiddles") == 3 * 3

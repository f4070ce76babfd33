"""The box passes' stages on pairs of lanes at 512 and 1024 points, thread by thread on the CPU: the twiddles they take from the
table, the force z chain of 512 points, the inverse y transforms."""
from test_layout_host import build_and_run


def test_pair_stages(tmp_path):
    out = build_and_run("host_pair512_check.cu", tmp_path / "pair512")
    assert out.count("rms rel error") == 4 and out.count("twiddles") == 2

"""The blocked layout's index map and the y passes' row offsets at every length that uses them, on the CPU."""
from test_layout_host import build_and_run


def test_index_maps_and_row_offsets(tmp_path):
    out = build_and_run("host_rows_check.cu", tmp_path / "rows_check")
    assert out.count("one-to-one") == 8 and out.count("rows consistent") == 11

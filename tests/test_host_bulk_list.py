"""The ensemble's bulk launches keep within the caller's blocks per SM:
tests/host_bulk_list.cu (bulk_list_blocks)."""
from test_host_headers import _build_and_run


def test_bulk_lists_keep_within_ctas_per_sm(tmp_path):
    out = _build_and_run(tmp_path, "host_bulk_list", "")
    assert "cases 224 failed 0" in out, out

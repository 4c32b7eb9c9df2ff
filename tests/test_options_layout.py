"""The options structure: a field added later lies where the compiler left a gap
before, so that programs built against the earlier header pass what they meant."""
import ctypes

from paper_1208_0274_gb300 import ae


def test_layout_and_choice():
    o = ae.ae_options_default()
    off = {k: getattr(ae.ae_options, k).offset for k, _ in ae.ae_options._fields_}
    assert ctypes.sizeof(ae.ae_options) == 88
    assert (off["tier_stats"], off["leaf_wide_auto"], off["workspace_limit"], off["leaf_wide_rows"]) == (48, 52, 56, 84)
    assert (o.leaf_wide_auto, o.leaf_wide_rows) == (1, 128)
    assert ae.make_options(leaf_wide_rows=128).leaf_wide_auto == 0
    assert ae.make_options(leaf_wide_rows=128, leaf_wide_auto=1).leaf_wide_auto == 1
    assert ae.make_options(leaf_delay=3).leaf_wide_auto == 1

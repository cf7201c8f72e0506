"""Device workspace of a solve by element type (fw_solve_plan, host only)."""
import pytest

import paper_2403_18619_gb300 as fw


def _bytes(n, bs, dtype):
    return fw.fw_solve_plan(n, fw.Options.default(bs=bs), sms=152, dtype=dtype)["workspace_bytes"]


@pytest.mark.parametrize("n", [700, 8192, 65536])
def test_only_filtered_tiles_have_16_bit_bounds(n):
    """fp64 in blocks of 64 keeps 16-bit bounds of its panels (two slots of two
    panels) and an exponent per round; int64 and blocks of 32 keep neither."""
    up = lambda b: (b + 255) // 256 * 256
    R = (n + 63) // 64
    assert _bytes(n, 64, fw.FW_F64) - _bytes(n, 64, fw.FW_I64) == \
        up(2 * R * 64 * 64 * 4) + up(R * 4)
    if n <= 32768:
        assert _bytes(n, 32, fw.FW_F64) == _bytes(n, 32, fw.FW_I64)

"""The peaks that bench.py compares solves with (CPU, with a stand-in for the
library): the loop over 16-bit keys where tiles may take it, since the 32-bit one
is half as fast and a solve above its "peak" says nothing."""
import types

import bench


def _fake():
    m = types.SimpleNamespace(FW_I32=0, FW_F32=1, FW_I64=2, FW_F64=3)
    m.fw_peak_probe = lambda dtype=0: (1e12 * (dtype + 1), 60.0, 2000.0)
    m.fw_peak_probe_keys16 = lambda: (4e13, 122.0, 2000.0)
    return m


def test_peak_of_the_loop_a_solve_takes():
    m = _fake()
    for dt in (m.FW_I32, m.FW_F64):
        rps, clk, mhz, name = bench.path_peak(m, dt)
        assert (rps, clk) == (4e13, 122.0) and "16" in name
    for dt in (m.FW_F32, m.FW_I64):
        rps, clk, mhz, name = bench.path_peak(m, dt)
        assert rps == 1e12 * (dt + 1) and "16" not in name

"""GPU test (-m gpu): the relaxation peak over 16-bit keys, two relaxations per
DPX instruction, is about twice the one over 32-bit keys."""
import pytest

from fwtest import fw

pytestmark = pytest.mark.gpu


def test_peak_probe_keys16():
    m = fw()
    rps, per_clk, mhz = m.fw_peak_probe_keys16()
    rps32, per_clk32, _ = m.fw_peak_probe(m.FW_I32)
    assert 300 <= mhz <= 2200 and rps > 1e12
    assert 1.6 * per_clk32 <= per_clk <= 2.1 * per_clk32

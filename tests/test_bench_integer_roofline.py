"""The benchmark's integer roofline of the FP64 waveform kernel (host only)."""
import pytest

import bench


def test_integer_roofline_arithmetic():
    # 29 multiply-adds per harmonic, 221 per sample besides
    assert bench.int_mad_model(20) == 29 * 20 + 221 == 801
    # 152 SMs x 4 sub-partitions x 32 lanes / 4 cycles x 2.07 GHz
    assert bench.INT_MAD_PEAK_T == pytest.approx(10.06848, rel=1e-12)
    # at 128 walkers x 2^21 in 30.1 ms: below the pipe's rate
    assert 0.6 < bench.int_mad_model(20) * 128 * 2 ** 21 / 30.1e-3 / 1e12 / bench.INT_MAD_PEAK_T < 1.0
    # the series it writes, 16 bytes, and the orbit records
    assert 16.0 < bench.K2_FIXED_DRAM_BYTES_PER_SAMPLE < 16.5

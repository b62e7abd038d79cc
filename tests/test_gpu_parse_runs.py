"""GPU tests of the compressor's parse where Dependency Elimination cuts nearly
every match to nothing: runs of one byte and short periods."""
import numpy as np
import pytest

import oracle

from test_gpu_tile import KiB, gmp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("n", [31, 512, 513, 2047, 2048, 2049, 2080, 70_001])
def test_streams_of_runs(gmp, n, byte_mode):  # noqa: F811
    rng = np.random.default_rng(n)
    for data in (np.zeros(n, np.uint8), np.resize(rng.integers(0, 256, 37).astype(np.uint8), n),
                 np.repeat(rng.integers(0, 256, n // 200 + 1).astype(np.uint8), 200)[:n]):
        for lazy in (False, True):
            s = gmp.compress_gpu(data, 64 * KiB, 16, 32 * KiB, de=True, byte_mode=byte_mode, lazy=lazy)
            rep = oracle.validate(s)
            assert rep["rc"] == 0 and rep["blocks_ok"] and rep["de_weak_ok"]
            assert np.array_equal(oracle.decompress(s), data)


def test_runs_take_no_longer_than_eight_times_ordinary_data(gmp):  # noqa: F811
    import datagen
    size = 1 << 20

    def parse_ms(data):
        times = []
        for _ in range(3):
            gmp.compress_gpu(data, 256 * KiB, 32, 32 * KiB, de=True)
            times.append(gmp.compress_gpu_times()["parse_ms"])
        return min(times)

    # one decision per position took 70 times as long
    assert parse_ms(np.zeros(size, np.uint8)) < 8 * parse_ms(datagen.csv_records(size, seed=3))

"""GPU tests of the entropy coder's CTA sizes (1024 to 128 threads per block, by
the number of blocks): valid streams on both sides of each step, and the time
of many small blocks."""
import numpy as np
import pytest

import datagen
import oracle

from test_gpu_tile import KiB, gmp, inputs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("rounds", [1, 2, 4])
def test_block_counts(gmp, rounds, byte_mode):  # noqa: F811
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n_blocks in (rounds * sms, rounds * sms + 1):
        for kind, block, n_sub in (("text", 997, 64), ("far", 3000, 3), ("zeros", 129, 16)):
            data = inputs(kind, n_blocks * block - 7, 100 + n_blocks)
            s = gmp.compress_gpu(data, block, n_sub, block, byte_mode=byte_mode)
            rep = oracle.validate(s)
            assert rep["rc"] == 0 and rep["offsets_ok"] and rep["blocks_ok"]
            assert byte_mode or (rep["kraft_ok"] and rep["lengths_ok"] and rep["subblocks_ok"])
            assert np.array_equal(oracle.decompress(s), data)


def test_many_small_blocks_are_coded_side_by_side(gmp):  # noqa: F811
    data = datagen.markov_text(16 << 20, seed=6, order=3)

    def encode_ms(block):
        times = []
        for _ in range(3):
            gmp.compress_gpu(data, block, 4, min(block, 32 * KiB))
            times.append(gmp.compress_gpu_times()["encode_ms"])
        return min(times)

    # 64 times as many trees; 30 times as long with one block on an SM at a time
    assert encode_ms(1 * KiB) < 12 * encode_ms(64 * KiB)

"""GPU test of the launch-shape tuner on batches whose blocks all run at once:
no shape that fills the SMs by half is kept for the larger batches to come."""
import numpy as np
import pytest

import datagen

from test_gpu_tile import KiB, gmp  # noqa: F401

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(600, method="thread")]


@pytest.mark.parametrize("byte_mode", [False, True])
def test_small_batches_keep_full_shapes(gmp, byte_mode):  # noqa: F811
    # 24 blocks: a CTA each when decoded, a pair of warps on 24 SMs when timed
    import torch
    ctx = gmp.Context(max_block_out=64 * KiB)
    data = datagen.csv_records(24 * 64 * KiB, seed=44)
    ds = gmp.DeviceStream(gmp.compress(data, 64 * KiB, 32, 32 * KiB, byte_mode=byte_mode))
    out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
    table = gmp.make_file_table([ds.file_desc(out)])
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    picked = {(t["warps_per_cta"], t["ctas_per_sm"]) for t in (ctx.autotune(table, 1, status) for _ in range(6))}
    assert all(w * c == 16 for w, c in picked), picked  # 16 blocks per SM, as many as fit
    assert int(status.item()) == 0 and np.array_equal(out.cpu().numpy(), data)
    ctx.close()

"""GPU tests of the decode kernel that gives a pair of warps to each block,
which launches of many blocks take: the data's bytes where a group of 64
records is halved (long matches, many far sources, long literal strings) or
written record by record, at odd record counts and unaligned outputs, and the
status of the kernel that keeps statistics on a corrupt block among good ones."""
import numpy as np
import pytest

from test_gpu_tile import KiB, check, ctx, gmp, inputs  # noqa: F401

pytestmark = pytest.mark.gpu

BLOCKS = 1000  # more than launches with a CTA per block take


def many(kind, block, seed):
    one = inputs(kind, 7 * block + 3, seed)
    return np.resize(one, BLOCKS * block - block // 2 - 1)


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("kind", ["text", "csv", "random", "zeros", "periods", "far"])
def test_kinds_of_data(gmp, ctx, kind, byte_mode):  # noqa: F811
    data = many(kind, 16 * KiB, 11)
    check(gmp, ctx, gmp.compress(data, 16 * KiB, 16, 16 * KiB, byte_mode=byte_mode), data)
    check(gmp, ctx, gmp.compress(data, 16 * KiB - 5, 33, 9000, de=True, byte_mode=byte_mode), data)


@pytest.mark.parametrize("block,max_match", [(1, 64), (3, 64), (131, 17), (5839, 64), (5841, 3)])
@pytest.mark.parametrize("byte_mode", [False, True])
def test_small_blocks(gmp, ctx, block, max_match, byte_mode):  # noqa: F811
    data = many("text", block, 12)
    check(gmp, ctx, gmp.compress(data, block, 3, 4096, max_match=max_match, byte_mode=byte_mode), data)


@pytest.mark.parametrize("byte_mode", [False, True])
def test_unaligned_output(gmp, ctx, byte_mode):  # noqa: F811
    import torch
    data = many("far", 20_000, 13)
    ds = gmp.DeviceStream(gmp.compress(data, 20_000, 16, 16 * KiB, byte_mode=byte_mode))
    base = torch.full((data.size + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.decompress_into(ds, base[1:1 + data.size], st)
    b = base.cpu().numpy()
    assert int(st.item()) == 0 and np.array_equal(b[1:1 + data.size], data)
    assert b[0] == 0xA5 and np.all(b[1 + data.size:] == 0xA5)


@pytest.mark.parametrize("byte_mode", [False, True])
def test_corrupt_block_among_good_ones(gmp, ctx, byte_mode):  # noqa: F811
    ref = gmp.Context(max_block_out=256 * KiB, collect_stats=True)
    data = many("csv", 4096, 14)
    s = gmp.compress(data, 4096, 4, 4096, byte_mode=byte_mode)
    rng = np.random.default_rng(15)
    lo, hi = (int(v) for v in s[64 + 8 * 500:64 + 8 * 502].view(np.uint64))
    failed = 0
    for _ in range(60):
        bad = s.copy()
        bad[int(rng.integers(lo + 8, hi))] ^= np.uint8(1 << int(rng.integers(0, 8)))
        try:
            ds = gmp.DeviceStream(bad)
        except gmp.GmpError:
            continue
        out_r, st_r = ref.decompress(ds)
        out, st = ctx.decompress(ds)
        assert (st == 0) == (st_r == 0), (st, st_r)
        failed += st != 0
        keep = np.ones(data.size, bool)
        keep[500 * 4096:501 * 4096] = st == 0
        assert np.array_equal(out.cpu().numpy()[keep], out_r.cpu().numpy()[keep])
    assert failed > 5
    ref.close()

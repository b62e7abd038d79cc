"""GPU tests of the status codes of damaged streams: the default kernels report
what the kernel of a forced resolution reports, the first damaged sub-block's
(or record's) failure, whichever lane or warp met it first."""
import numpy as np
import pytest

import datagen
import oracle

from test_gpu_tile import KiB, ctx, gmp  # noqa: F401

pytestmark = pytest.mark.gpu


def flips(s, lo, hi, table, seed, n):
    """n copies of s with one bit flipped in [lo, hi), one in three in [lo, table)."""
    rng = np.random.default_rng(seed)
    for k in range(n):
        bad = s.copy()
        bad[int(rng.integers(lo, table if k % 3 == 0 else hi))] ^= np.uint8(1 << int(rng.integers(0, 8)))
        yield bad


def compare(gmp, ctx, streams):  # noqa: F811
    ref = gmp.Context(max_block_out=256 * KiB, resolve="mrr")
    seen = set()
    for bad in streams:
        try:
            ds = gmp.DeviceStream(bad)
        except gmp.GmpError:
            continue
        st, want = ctx.decompress(ds)[1], ref.decompress(ds)[1]
        assert st == want, (gmp.STATUS_NAMES[st], gmp.STATUS_NAMES[want])
        seen.add(st)
    ref.close()
    return seen


@pytest.mark.parametrize("n_sub", [1, 16, 32, 64])
def test_huffman_block(gmp, ctx, n_sub):  # noqa: F811
    data = datagen.markov_text(60_000, seed=31 + n_sub, order=3)
    s = oracle.compress(data, oracle.params(64 * KiB, n_sub, 8 * KiB))
    lo = int(s[64:72].view(np.uint64)[0])
    # with more than 32 sub-blocks, the bits of one sub-block at a time (a
    # damaged table fails many, and the other kernel takes 32 of them at once)
    first = lo if n_sub <= 32 else lo + (192 + 12 * n_sub + 15) // 16 * 16
    seen = compare(gmp, ctx, flips(s, first, s.size - 17, first + 400, n_sub, 500))
    assert {oracle.BITSTREAM, oracle.BAD_OFFSET, oracle.OUTPUT_OVERRUN} <= seen


def test_byte_block(gmp, ctx):  # noqa: F811
    data = datagen.markov_text(60_000, seed=31, order=3)
    s = oracle.compress(data, oracle.params(64 * KiB, 1, 8 * KiB, byte_mode=True))
    lo = int(s[64:72].view(np.uint64)[0])
    streams = list(flips(s, lo, s.size - 17, lo + 400, 3, 500))
    n_seq = int(s[lo:lo + 4].view(np.uint32)[0])
    for k in np.linspace(0, n_seq - 1, 40).astype(int):  # a match code without a length
        bad = s.copy()
        bad[lo + 16 + 4 * k:lo + 20 + 4 * k].view(np.uint32)[0] |= 63 << 10
        streams.append(bad)
    assert {oracle.CORRUPT_SYMBOL, oracle.BAD_OFFSET, oracle.OUTPUT_OVERRUN} <= compare(gmp, ctx, streams)


@pytest.mark.parametrize("byte_mode", [False, True])
def test_one_block_of_many(gmp, ctx, byte_mode):  # noqa: F811
    # 1000 blocks: a pair of warps each
    data = np.resize(datagen.csv_records(7 * 4096, seed=14), 1000 * 4096 - 2049)
    s = gmp.compress(data, 4096, 4, 4096, byte_mode=byte_mode)
    lo, hi = (int(v) for v in s[64 + 8 * 500:64 + 8 * 502].view(np.uint64))
    assert len(compare(gmp, ctx, flips(s, lo + 8, hi, lo + 250, 15, 200))) > 2


@pytest.mark.parametrize("copies", [1, 1000])
@pytest.mark.parametrize("order", [0, 1])
def test_first_damaged_sub_block_decides(gmp, ctx, order, copies):  # noqa: F811
    # two sub-blocks whose stated sizes are wrong by a bit and by a byte of
    # output: the lower one's failure is the status
    import torch
    data = datagen.markov_text(60_000, seed=5, order=3)
    s = oracle.compress(data, oracle.params(64 * KiB, 16, 8 * KiB))
    t = int(s[64:72].view(np.uint64)[0]) + 192
    table = s[t:t + 12 * 16].view(np.uint32).reshape(16, 3).copy()
    bits_at, out_at = (3, 9) if order == 0 else (9, 3)
    # (a bit and a byte moved to the sub-block after, so that the totals stay)
    table[bits_at, 0] += 1
    table[bits_at + 1, 0] -= 1
    table[out_at, 1] += 1
    table[out_at + 1, 1] -= 1
    s[t:t + 12 * 16] = np.ascontiguousarray(table).view(np.uint8).reshape(-1)
    ds = gmp.DeviceStream(s)
    out = torch.zeros(copies * 60_000 + 16 * copies, dtype=torch.uint8, device="cuda")
    st = torch.zeros(copies, dtype=torch.int32, device="cuda")
    files = gmp.make_file_table([ds.file_desc(out[i * 60_016:i * 60_016 + 60_000]) for i in range(copies)])
    ctx.decompress_batch(files, copies, st)
    assert st.cpu().unique().tolist() == [oracle.BITSTREAM if order == 0 else oracle.OUTPUT_OVERRUN]

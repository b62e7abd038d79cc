"""GPU tests of blocks of long literal strings, which take groups of fewer records
(Byte blocks) or records of up to seven literals (Huffman blocks): the oracle's
bytes for every kind of literal length and distance, decoded by a CTA per block
and (more blocks) by a pair of warps per block, at aligned and unaligned
outputs, damaged blocks among them, and the time beside that of text."""
import numpy as np
import pytest

import oracle

from test_gpu_tile import KiB, ctx, gmp  # noqa: F401

pytestmark = pytest.mark.gpu

PAIRS = 1000  # more blocks than launches with a CTA per block take


def tokens(seed, n, lits, dists):
    """n sequences with literal lengths and distances drawn from the given
    values; two in three distances reach at most 40 bytes back."""
    rng = np.random.default_rng(seed)
    ll = rng.choice(lits, n).astype(np.uint32)
    ml = rng.integers(3, 65, n).astype(np.uint32)
    ml[rng.random(n) < 0.2] = 0
    ml[-1] = 0
    ll[0] = max(int(ll[0]), 1)
    at = np.cumsum(ll.astype(np.int64)) + np.concatenate([[0], np.cumsum(ml.astype(np.int64))[:-1]])
    near = np.minimum(rng.integers(1, 41, n), at)
    dist = np.where(rng.random(n) < 0.66, near, np.minimum(rng.choice(dists, n), at)).astype(np.uint32)
    dist[ml == 0] = 0
    return ll, ml, dist, rng.integers(0, 256, int(ll.sum())).astype(np.uint8)


def decode(gmp, ctx, stream, data, copies, offset):  # noqa: F811
    """The stream `copies` times in one batched launch: the statuses, whether
    every output is `data`, and whether nothing was written between them."""
    import torch
    ds = gmp.DeviceStream(stream)
    size, stride = data.size, (data.size + 63) // 16 * 16
    out = torch.full((copies * stride + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    st = torch.zeros(copies, dtype=torch.int32, device="cuda")
    table = gmp.make_file_table([ds.file_desc(out[offset + i * stride:offset + i * stride + size])
                                 for i in range(copies)])
    ctx.decompress_batch(table, copies, st)
    rows = out[offset:offset + copies * stride].view(copies, stride)
    want = torch.from_numpy(data).cuda()
    return st.cpu().numpy(), bool((rows[:, :size] == want).all()), bool((rows[:, size:] == 0xA5).all())


LENGTHS = {"few": [0, 1, 2, 5, 9], "mean 12": [0, 8, 12, 17, 24], "mean 31": [15, 16, 31, 32, 63],
           "mean 100": [0, 1, 100, 200, 255], "long": [500, 511, 512, 513, 1023], "only": [1023],
           "some": [0, 1, 2, 3, 4, 5, 6, 1000]}


@pytest.mark.parametrize("copies", [1, 40, PAIRS])
@pytest.mark.parametrize("kind", list(LENGTHS))
def test_literal_lengths(gmp, ctx, kind, copies):  # noqa: F811
    for seed, n in ((1, 2), (2, 63), (3, 65), (4, 700)):
        ll, ml, dist, lits = tokens(seed, n, LENGTHS[kind], [1, 2, 31, 32, 33, 127, 128, 1000, 1040, 2500, 30_000])
        s = gmp.encode_tokens(ll, ml, dist, lits, byte_mode=True)
        data = oracle.lz77_decode(ll, ml, dist, lits)
        for offset in (0, 16, 3):
            st, same, guard = decode(gmp, ctx, s, data, copies, offset)
            assert not st.any() and same and guard, (n, offset)


@pytest.mark.parametrize("copies", [1, PAIRS])
@pytest.mark.parametrize("kind", ["mean 31", "long", "some"])
def test_damaged_records(gmp, ctx, kind, copies):  # noqa: F811
    ll, ml, dist, lits = tokens(9, 300, LENGTHS[kind], [1, 40, 1000, 5000])
    s = gmp.encode_tokens(ll, ml, dist, lits, byte_mode=True)
    data = oracle.lz77_decode(ll, ml, dist, lits)
    at = int(s[64:72].view(np.uint64)[0]) + 16
    rng = np.random.default_rng(3)
    failed = 0
    for _ in range(25):
        bad = s.copy()
        bad[at + int(rng.integers(0, 4 * 300))] ^= np.uint8(1 << int(rng.integers(0, 8)))
        want = oracle.decompress_status(bad)
        st, same, guard = decode(gmp, ctx, bad, data if want else oracle.decompress(bad), copies, 0)
        assert ((st != 0) == (want != 0)).all() and guard and (want != 0 or same)
        failed += want != 0
    assert failed > 5


HUFFMAN = {"3 to 9": [3, 4, 5, 6, 7, 8, 9], "around 14": [12, 13, 14, 15, 16], "mean 31": [15, 16, 31, 32, 63],
           "long": [255, 256, 257, 1023, 5000], "some": [0, 1, 2, 3, 4, 5, 6, 1000]}


def huffman_stream(gmp, kind, seed, n, n_sub):  # noqa: F811
    ll, ml, dist, lits = tokens(seed, n, HUFFMAN[kind], [1, 2, 31, 33, 1000, 2500, 30_000])
    ml = np.maximum(ml, 3)  # every sequence but the last has a match
    ml[-1] = 0
    at = np.cumsum(ll.astype(np.int64)) + np.concatenate([[0], np.cumsum(ml.astype(np.int64))[:-1]])
    dist = np.where(ml > 0, np.clip(dist, 1, np.minimum(at, 32768)), 0).astype(np.uint32)
    if seed % 2:
        lits = np.minimum(lits, 40 + lits % 30)  # shorter codes: lookups of two literals
    return gmp.encode_tokens(ll, ml, dist, lits, n_sub=n_sub), oracle.lz77_decode(ll, ml, dist, lits)


@pytest.mark.parametrize("copies", [1, 200, PAIRS])
@pytest.mark.parametrize("kind", list(HUFFMAN))
def test_huffman_literal_lengths(gmp, ctx, kind, copies):  # noqa: F811
    for seed, n, n_sub in ((1, 2, 1), (2, 40, 3), (3, 65, 33), (4, 700, 64), (5, 900, 32), (6, 30, 16)):
        s, data = huffman_stream(gmp, kind, seed, n, n_sub)
        if data.size > 256 * KiB:  # what the context's blocks may hold
            continue
        for offset in (0, 16, 3):
            st, same, guard = decode(gmp, ctx, s, data, copies, offset)
            assert not st.any() and same and guard, (seed, offset)


@pytest.mark.parametrize("copies", [1, PAIRS])
@pytest.mark.parametrize("kind", ["3 to 9", "mean 31", "some"])
def test_damaged_huffman_blocks(gmp, ctx, kind, copies):  # noqa: F811
    s, data = huffman_stream(gmp, kind, 7, 300, 16)
    lo = int(s[64:72].view(np.uint64)[0])
    rng = np.random.default_rng(4)
    failed = 0
    for k in range(40):
        bad = s.copy()
        bad[int(rng.integers(lo, lo + 400 if k % 3 == 0 else s.size - 17))] ^= np.uint8(1 << int(rng.integers(0, 8)))
        want = oracle.decompress_status(bad)
        try:
            st, same, guard = decode(gmp, ctx, bad, data if want else oracle.decompress(bad), copies, 0)
        except gmp.GmpError:
            continue
        assert ((st != 0) == (want != 0)).all() and guard and (want != 0 or same)
        failed += want != 0
    assert failed > 5


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("block,n_blocks", [(16 * KiB, 1100), (64 * KiB, 700)])  # a pair of warps, a CTA per block
def test_time_beside_text(gmp, ctx, block, n_blocks, byte_mode):  # noqa: F811
    import torch

    import datagen

    def microseconds(data):
        ds = gmp.DeviceStream(gmp.compress(np.resize(data, n_blocks * block), block, byte_mode=byte_mode, chain_depth=16))
        out = torch.zeros(n_blocks * block, dtype=torch.uint8, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.decompress_into(ds, out, st)
            b.record()
            torch.cuda.synchronize()
            times.append(1e3 * a.elapsed_time(b))
        assert int(st.item()) == 0
        return min(times[2:])

    rng = np.random.default_rng(1)
    rows = rng.integers(0, 256, (8 << 10, 40)).astype(np.uint8)  # 31 literals, a copy of 9 bytes from 20 rows back
    for i in range(20, len(rows)):
        rows[i, 31:] = rows[i - 20, 3:12]
    # Byte blocks: 2.6 and 4 times as long when such groups were written record after
    # record.  Huffman blocks have three times as many codes per byte.
    assert microseconds(rows.reshape(-1)) < (1.5 if byte_mode else 2.5) * microseconds(datagen.markov_text(1 << 20, seed=2, order=3))

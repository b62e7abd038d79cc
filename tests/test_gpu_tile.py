"""GPU tests of the default decode kernel (contexts without statistics or a
forced resolution): the oracle's bytes at the edges of its tiles, groups,
window and staging, and the status of the kernel that keeps statistics on
corrupt streams."""
import numpy as np
import pytest

import datagen
import oracle

pytestmark = pytest.mark.gpu

KiB, MiB = 1 << 10, 1 << 20


@pytest.fixture(scope="module")
def gmp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1606_00519_gb300 import _native
    _native.build()
    import paper_1606_00519_gb300 as g
    return g


@pytest.fixture(scope="module")
def ctx(gmp):
    c = gmp.Context(max_block_out=256 * KiB)
    yield c
    c.close()


def check(gmp, ctx, stream, data):
    out, status = ctx.decompress(gmp.DeviceStream(stream))
    got = out.cpu().numpy()
    assert status == 0, gmp.STATUS_NAMES.get(status, status)
    if not np.array_equal(got, data):
        bad = np.flatnonzero(got != data)
        raise AssertionError(f"{bad.size} of {data.size} bytes differ, first at {int(bad[0])}")


def inputs(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "text":
        return datagen.markov_text(n, seed=seed, order=3)
    if kind == "csv":
        return datagen.csv_records(n, seed=seed)
    if kind == "random":  # literals only, at 8 bits and more
        return rng.integers(0, 256, n).astype(np.uint8)
    if kind == "zeros":  # distance 1
        return np.zeros(n, np.uint8)
    if kind == "periods":  # overlapping copies of every short period
        parts, p = [], 1
        while sum(map(len, parts)) < n:
            parts.append(np.resize(rng.integers(0, 256, p).astype(np.uint8), 300))
            p = p % 40 + 1
        return np.concatenate([np.zeros(0, np.uint8), *parts])[:n]
    # runs of literals of up to 4000 bytes between repeats from far back
    base = rng.integers(0, 256, 30_000).astype(np.uint8)
    parts = [base]
    while sum(map(len, parts)) < n:
        parts.append(rng.integers(0, 256, int(rng.integers(1, 4000))).astype(np.uint8))
        at = int(rng.integers(0, 29_000))
        parts.append(base[at:at + int(rng.integers(3, 900))])
    return np.concatenate(parts)[:n]


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("kind", ["text", "csv", "random", "zeros", "periods", "far"])
def test_kinds_of_data(gmp, ctx, kind, byte_mode):
    data = inputs(kind, 700_001, 3)
    for de in (False, True):
        check(gmp, ctx, gmp.compress(data, 256 * KiB, 32, 32 * KiB, de=de, byte_mode=byte_mode), data)
        check(gmp, ctx, gmp.compress(data, 100_000, 33, 20_000, de=de, byte_mode=byte_mode), data)


@pytest.mark.parametrize("size", [0, 1, 2, 15, 16, 17, 31, 32, 33, 127, 128, 129, 511, 512, 513, 4095, 6287, 6288, 6289,
                                  65535, 65537])
@pytest.mark.parametrize("byte_mode", [False, True])
def test_sizes(gmp, ctx, size, byte_mode):
    for kind in ("text", "periods"):
        data = inputs(kind, size, size + 1)
        check(gmp, ctx, gmp.compress(data, 64 * KiB, 16, 8 * KiB, byte_mode=byte_mode), data)


@pytest.mark.parametrize("n_sub,cwl", [(1, 12), (3, 12), (31, 10), (32, 9), (33, 12), (64, 11)])
def test_sub_block_counts_and_code_lengths(gmp, ctx, n_sub, cwl):
    data = inputs("text", 400_000, n_sub)
    check(gmp, ctx, gmp.compress(data, 128 * KiB, n_sub, 32 * KiB, cwl=cwl), data)
    rng = np.random.default_rng(n_sub)  # skewed literals: codes of every length up to cwl
    data = np.minimum(rng.geometric(0.35, 300_000) * 7 + rng.integers(0, 3, 300_000), 255).astype(np.uint8)
    check(gmp, ctx, gmp.compress(data, 128 * KiB, n_sub, 32 * KiB, cwl=cwl), data)


@pytest.mark.parametrize("block,window,max_match", [(1000, 1, 64), (4093, 4096, 3), (12345, 257, 17), (16, 8, 64)])
def test_small_blocks_and_windows(gmp, ctx, block, window, max_match):
    data = inputs("text", 50_000, 8)
    for byte_mode in (False, True):
        check(gmp, ctx, gmp.compress(data, block, 4, window, max_match=max_match, byte_mode=byte_mode), data)


@pytest.mark.parametrize("block", [256 * KiB + 16, 1 * MiB])
def test_large_blocks(gmp, block):
    c = gmp.Context(max_block_out=1 * MiB)
    data = np.concatenate([inputs("text", 1_200_000, 21), inputs("zeros", 300_000, 0), inputs("far", 900_000, 5)])
    for byte_mode in (False, True):
        check(gmp, c, gmp.compress(data, block, 64, 32 * KiB, byte_mode=byte_mode), data)
    c.close()


@pytest.mark.parametrize("offset", [1, 8, 16])
def test_output_alignment_and_guard_bytes(gmp, ctx, offset):
    import torch
    data = inputs("far", 300_001, 4)
    for byte_mode in (False, True):
        ds = gmp.DeviceStream(gmp.compress(data, 64 * KiB, 16, 32 * KiB, byte_mode=byte_mode))
        base = torch.full((data.size + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        ctx.decompress_into(ds, base[offset:offset + data.size], st)
        b = base.cpu().numpy()
        assert int(st.item()) == 0 and np.array_equal(b[offset:offset + data.size], data)
        assert np.all(b[:offset] == 0xA5) and np.all(b[offset + data.size:] == 0xA5)


@pytest.mark.parametrize("m", [1, 2, 8, 32])
@pytest.mark.parametrize("byte_mode", [False, True])
def test_nested_references(gmp, ctx, m, byte_mode):
    ts = datagen.nesting_tokens(seed=400 + m, m=m, n_inst=32 * 50)
    s = gmp.encode_tokens(ts.lit_len, ts.mlen, ts.off, ts.lits, n_sub=32, byte_mode=byte_mode)
    check(gmp, ctx, s, oracle.lz77_decode(ts.lit_len, ts.mlen, ts.off, ts.lits))


@pytest.mark.parametrize("n_blocks", [1, 5, 300, 700, 1500, 3200])
def test_block_counts(gmp, n_blocks):
    # from one block to more blocks than the GPU runs at once, alone and in a
    # batch of two files
    import torch
    c = gmp.Context(max_block_out=16 * KiB)
    data = inputs("csv", n_blocks * 16 * KiB - 5, n_blocks)
    for byte_mode in (False, True):
        s = gmp.compress(data, 16 * KiB, 16, 16 * KiB, byte_mode=byte_mode)
        check(gmp, c, s, data)
        ds = gmp.DeviceStream(s)
        outs = [torch.zeros(data.size, dtype=torch.uint8, device="cuda") for _ in range(2)]
        st = torch.zeros(2, dtype=torch.int32, device="cuda")
        c.decompress_batch(gmp.make_file_table([ds.file_desc(o) for o in outs]), 2, st)
        assert st.cpu().tolist() == [0, 0]
        assert all(np.array_equal(o.cpu().numpy(), data) for o in outs)
        got, status = c.decompress_host(s)
        assert status == 0 and np.array_equal(got, data)
    c.close()


@pytest.mark.parametrize("byte_mode", [False, True])
def test_corrupt_streams(gmp, ctx, byte_mode):
    # single-block streams, so that one status is the first in both kernels
    ref = gmp.Context(max_block_out=256 * KiB, collect_stats=True)
    data = inputs("text", 60_000, 31)
    s = oracle.compress(data, oracle.params(64 * KiB, 1 if byte_mode else 16, 8 * KiB, byte_mode=byte_mode))
    rng = np.random.default_rng(77)
    lo = int(s[64:72].view(np.uint64)[0])
    seen = set()
    for k in range(150):
        bad = s.copy()
        i = int(rng.integers(lo, lo + 400 if k % 3 == 0 else s.size - 17))
        bad[i] ^= np.uint8(1 << int(rng.integers(0, 8)))
        try:
            ds = gmp.DeviceStream(bad)
        except gmp.GmpError:
            continue
        out_r, st_r = ref.decompress(ds)
        out, st = ctx.decompress(ds)
        assert (st == 0) == (st_r == 0) == (oracle.decompress_status(bad) == 0), (i, st, st_r)
        seen.add(st)
        if st == 0:
            assert np.array_equal(out.cpu().numpy(), out_r.cpu().numpy())
    assert len(seen) > 2
    bad = s.copy()
    bad[16:20] = np.frombuffer(np.uint32(2).tobytes(), np.uint8)  # header window = 2
    assert ctx.decompress(gmp.DeviceStream(bad))[1] == oracle.BAD_OFFSET
    ref.close()

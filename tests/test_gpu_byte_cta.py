"""GPU tests of Byte blocks in the kernel that gives a CTA to each block: the
data's bytes where literal strings outgrow a wave, or a whole group is written
record by record, between ordinary waves; every stream new, so that its
literals come from device memory, alone and mixed with Huffman files."""
import numpy as np
import pytest

import datagen

from test_gpu_tile import KiB, ctx, gmp  # noqa: F401

pytestmark = pytest.mark.gpu


def waves(n, seed):
    """Text with runs of random bytes between: of a few bytes per record (two
    or three waves where one would do), and of up to 4000 (whole groups)."""
    rng = np.random.default_rng(seed)
    text = datagen.markov_text(n, seed=seed, order=3)
    parts, used = [], 0
    while used < n:
        kind, size = int(rng.integers(0, 4)), int(rng.integers(200, 6000))
        part = text[used:used + size]
        if kind == 1:
            part = part.copy()
            part[rng.integers(0, part.size, part.size // 12 + 1)] = rng.integers(0, 256, part.size // 12 + 1)
        elif kind == 2:
            part = rng.integers(0, 256, min(size, 4000)).astype(np.uint8)
        elif kind == 3:
            # records of 40 literals and a match: 64 of them make a group for
            # one warp alone
            lits = rng.integers(0, 256, (70, 40)).astype(np.uint8)
            part = np.concatenate([lits, np.tile(text[used:used + 1], (70, 8))], axis=1).reshape(-1)
        parts.append(part)
        used += part.size
    return np.concatenate(parts)[:n]


@pytest.mark.parametrize("n_blocks", [1, 8, 200])  # 16 warps per block (200: 8 warps)
@pytest.mark.parametrize("size", [4093, 70_000])
def test_new_streams(gmp, ctx, n_blocks, size):  # noqa: F811
    import torch
    for seed in range(24 if n_blocks < 200 else 3):
        data = np.resize(waves(min(n_blocks, 8) * size, seed), n_blocks * size)
        ds = gmp.DeviceStream(gmp.compress(data, size, byte_mode=True, de=seed % 2 == 1))
        out = torch.full((data.size,), 0xA5, dtype=torch.uint8, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        ctx.decompress_into(ds, out, st)
        assert int(st.item()) == 0 and np.array_equal(out.cpu().numpy(), data)


def test_mixed_files(gmp, ctx):  # noqa: F811
    # more blocks than CTAs at once, so that a CTA goes from a Byte block to a
    # Huffman block and back
    import torch
    datas = [waves(60_000 + 9_000 * i, 100 + i) for i in range(30)]
    streams = [gmp.DeviceStream(gmp.compress(d, 9_000, 16, 9_000, byte_mode=i % 2 == 0)) for i, d in enumerate(datas)]
    assert 456 < sum(s.n_blocks for s in streams) < 798
    outs = [torch.full((d.size,), 0xA5, dtype=torch.uint8, device="cuda") for d in datas]
    st = torch.zeros(len(datas), dtype=torch.int32, device="cuda")
    for pick in (slice(0, 30), slice(0, 20), slice(7, 21)):
        n = len(datas[pick])
        for o in outs:
            o.fill_(0xA5)
        ctx.decompress_batch(gmp.make_file_table([s.file_desc(o) for s, o in zip(streams[pick], outs[pick])]), n, st)
        assert st[:n].cpu().tolist() == [0] * n
        assert all(np.array_equal(o.cpu().numpy(), d) for o, d in zip(outs[pick], datas[pick]))

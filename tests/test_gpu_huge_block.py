"""GPU test of the compressor with a block of more than 2^32 coded bits: every
sub-block's codes stand where the block's sub-block table puts them."""
import numpy as np
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(600, method="thread")]

K = 64


@pytest.fixture(scope="module")
def gmp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1606_00519_gb300 import _native
    _native.build()
    import paper_1606_00519_gb300 as g
    return g


def code_table(lens):
    """{(length, code with its first bit lowest): symbol} of canonical lengths."""
    table, code = {}, 0
    for length in range(1, 13):
        for sym in np.flatnonzero(lens == length):
            table[length, int(f"{code:0{length}b}"[::-1], 2)] = int(sym)
            code += 1
        code <<= 1
    return table


def distance_bits(sym):
    """(base, extra bits) of an offset symbol."""
    extra = 0 if sym < 4 else (sym >> 1) - 1
    return (sym + 1 if sym < 4 else ((2 | (sym & 1)) << extra) + 1), extra


def test_sub_blocks_past_2_to_32_bits(gmp):
    n = 540 << 20
    data = np.random.default_rng(5).integers(0, 1 << 64, n // 8, dtype=np.uint64).view(np.uint8)
    s = gmp.compress_gpu(data, block_size=n, n_sub=K)
    at = int(s[64:72].view(np.uint64)[0])  # the only block
    nib = np.stack([s[at + 8:at + 192] & 15, s[at + 8:at + 192] >> 4], 1).reshape(-1)
    lits, offs = code_table(nib[:319]), code_table(nib[320:350])
    sizes = s[at + 192:at + 192 + 12 * K].view(np.uint32).reshape(K, 3).astype(np.int64)
    bit, out = (np.concatenate([[0], np.cumsum(sizes[:, i])]) for i in (0, 1))
    assert bit[-1] > 1 << 32 and out[-1] == n
    base = at + (192 + 12 * K + 15) // 16 * 16
    for j in range(K):
        lo = base + int(bit[j]) // 8
        bits = np.unpackbits(s[lo:lo + 1000], bitorder="little")[int(bit[j]) % 8:].tolist()
        p, o = 0, int(out[j])

        def code(table):
            nonlocal p
            v = 0
            for length in range(1, 13):
                v |= bits[p] << (length - 1)
                p += 1
                if (length, v) in table:
                    return table[length, v]
            raise AssertionError("no code")

        while p < 7000:  # a literal is the input's byte; a match repeats what lies its distance before
            sym = code(lits)
            if sym < 256:
                assert sym == data[o], (j, o)
                o += 1
            else:
                length = sym - 254
                first, extra = distance_bits(code(offs))
                dist = first + sum(b << i for i, b in enumerate(bits[p:p + extra]))
                p += extra
                assert np.array_equal(data[o:o + length], data[o - dist:o - dist + length]), (j, o)
                o += length

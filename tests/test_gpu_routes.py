"""GPU tests of what decides between the decode kernels: every launch shape of
the pair of warps per block, block counts at and around the limits of the CTA
per block (also where the device chooses, by the first stream's format), forced
resolutions without statistics, and a wait for input that runs out in the pair
kernel, whose second warp must follow the first."""
import time

import numpy as np
import pytest

from test_gpu_tile import KiB, gmp, inputs  # noqa: F401

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(600, method="thread")]

BLOCK = 4 * KiB


def stream(gmp, kind, n_blocks, byte_mode, de=False):  # noqa: F811
    data = np.resize(inputs(kind, 40 * BLOCK + 77, 9), n_blocks * BLOCK - 5)
    return data, gmp.compress(data, BLOCK, 8, BLOCK, de=de, byte_mode=byte_mode)


def check_all_calls(gmp, c, data, s):  # noqa: F811
    import torch
    ds = gmp.DeviceStream(s)
    out, st = c.decompress(ds)
    assert st == 0 and np.array_equal(out.cpu().numpy(), data)
    outs = [torch.zeros(data.size, dtype=torch.uint8, device="cuda") for _ in range(2)]
    sts = torch.zeros(2, dtype=torch.int32, device="cuda")
    c.decompress_batch(gmp.make_file_table([ds.file_desc(o) for o in outs]), 2, sts)
    assert sts.cpu().tolist() == [0, 0] and all(np.array_equal(o.cpu().numpy(), data) for o in outs)
    got, st = c.decompress_host(s)
    assert st == 0 and np.array_equal(got, data)
    got, sts = c.decompress_from_host_batch([s])
    assert sts == [0] and np.array_equal(got[0].cpu().numpy(), data)


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("shape", [(1, 0), (2, 0), (3, 0), (4, 0), (8, 0), (16, 0), (1, 1), (4, 2), (5, 1)])
def test_shapes_of_many_blocks(gmp, shape, byte_mode):  # noqa: F811
    data, s = stream(gmp, "far" if byte_mode else "csv", 2000, byte_mode)
    c = gmp.Context(max_block_out=BLOCK, warps_per_cta=shape[0], ctas_per_sm=shape[1])
    check_all_calls(gmp, c, data, s)
    c.set_launch(4, 0)
    check_all_calls(gmp, c, data, s)
    c.close()


@pytest.mark.parametrize("byte_mode", [False, True])
@pytest.mark.parametrize("of", [1.0, 3.0, 5.25, 6.0, 7.5, 12.0])  # blocks per SM at the limits
def test_limits(gmp, of, byte_mode):  # noqa: F811
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c = gmp.Context(max_block_out=BLOCK)
    for n in (int(of * sms) - 1, int(of * sms), int(of * sms) + 1):
        check_all_calls(gmp, c, *stream(gmp, "text", n, byte_mode))
    c.close()


@pytest.mark.parametrize("n", [100, 399, 430, 456, 457])
@pytest.mark.parametrize("byte_first", [False, True])
def test_mixed_batches(gmp, byte_first, n):  # noqa: F811
    # two files of n blocks, of both formats: the first one's decides the limit
    import torch
    made = [stream(gmp, "csv", n, byte_first), stream(gmp, "csv", n, not byte_first, de=True)]
    c = gmp.Context(max_block_out=BLOCK)
    dss = [gmp.DeviceStream(s) for _, s in made]
    outs = [torch.zeros(d.size, dtype=torch.uint8, device="cuda") for d, _ in made]
    st = torch.zeros(2, dtype=torch.int32, device="cuda")
    table = gmp.make_file_table([ds.file_desc(o) for ds, o in zip(dss, outs)])
    g = c.batch_graph(table, 2, st)
    for launch in (lambda: c.decompress_batch(table, 2, st), g.launch, g.launch):
        for o in outs:
            o.zero_()
        launch()
        assert st.cpu().tolist() == [0, 0]
        assert all(np.array_equal(o.cpu().numpy(), d) for o, (d, _) in zip(outs, made))
    g.close()
    c.close()


@pytest.mark.parametrize("resolve", ["mrr", "sc"])
@pytest.mark.parametrize("byte_mode", [False, True])
def test_forced_resolution_without_statistics(gmp, byte_mode, resolve):  # noqa: F811
    for n, shape in ((3, 0), (300, 8), (3300, 0)):
        c = gmp.Context(max_block_out=BLOCK, resolve=resolve, warps_per_cta=shape)
        check_all_calls(gmp, c, *stream(gmp, "periods", n, byte_mode, de=n == 300))
        c.close()


@pytest.mark.parametrize("byte_mode", [False, True])
def test_input_wait_runs_out_in_the_pair_kernel(gmp, byte_mode):  # noqa: F811
    # a flag dropped on the host: the blocks of that piece are skipped, the file
    # reports it, the other file is decoded and the context stays usable
    made = [stream(gmp, "csv", 1500, byte_mode), stream(gmp, "text", 600, byte_mode)]
    streams = [s for _, s in made]
    c = gmp.Context(max_block_out=BLOCK)
    c.set_input_wait(200)
    for call in (c.decompress_host_batch, c.decompress_from_host_batch):
        for piece in (0, 3):
            c.debug_drop_input_flag(piece)
            t0 = time.perf_counter()
            outs, sts = call(streams)
            assert time.perf_counter() - t0 < 5.0
            assert gmp.STATUS_NAMES[sts[0]] == "INPUT_TIMEOUT"
        outs, sts = call(streams)
        assert sts == [0, 0]
        for o, (d, _) in zip(outs, made):
            assert np.array_equal(o if isinstance(o, np.ndarray) else o.cpu().numpy(), d)
    c.close()

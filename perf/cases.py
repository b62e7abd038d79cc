"""The work this package does for its users, as measurable cases: decoding on the
device (one stream, a batch, many files in one graph launch), decoding from and
to host memory, and compressing on the GPU.

Text and records stand for the two kinds of data the package is used on: order-3
Markov text (about 2.7 times compressible) and CSV rows of ids, prices, dates and
categories (about 3 times).  Streams are written by the host compressor with its
defaults unless a case says otherwise.  A case is a dict:

  op      "stream"     one stream resident on the device, one decode call
          "batch"      streams of the same data in MRR and DE mode, one batched call
          "files"      files of 4 KiB - 16 MiB (log-uniform), both kinds and modes,
                       one CUDA graph launch
          "from_host"  stream in pinned host memory, output left on the device
          "host"       stream and output in pinned host memory
          "compress"   host buffer in, host stream out, all steps on the GPU
  data    "text" or "csv";  bytes: decompressed size (per stream)
  de      Dependency Elimination;  byte_mode: byte-level blocks without Huffman coding
  block, n_sub, window: the stream format's parameters
"""
import datetime
import math
import random

import numpy as np
import torch

import paper_1606_00519_gb300 as gmp

KiB, MiB = 1 << 10, 1 << 20
FILE_MIN, FILE_MAX = 4 * KiB, 16 * MiB


def _case(op, data, size, de=False, byte_mode=False, block=256 * KiB, n_sub=32, window=32 * KiB, **kw):
    return dict(kw, op=op, data=data, bytes=size, de=de, byte_mode=byte_mode, block=block, n_sub=n_sub, window=window)


def listed():
    return [
        # one small file: a single block, pure latency
        _case("stream", "text", 16 * KiB, name="stream_text_16k"),
        # a small stream of small blocks (64 KiB, 16 sub-blocks, 8 KiB window)
        _case("stream", "text", 1 * MiB, block=64 * KiB, n_sub=16, window=8 * KiB, name="stream_text_1m"),
        # an ordinary file, its size no multiple of anything
        _case("stream", "csv", 16 * MiB + 12345, de=True, name="stream_csv_16m_de"),
        # a larger one, fewer blocks than the GPU runs at once
        _case("stream", "text", 64 * MiB, name="stream_text_64m"),
        # byte-level blocks, for users who want speed over ratio
        _case("stream", "csv", 128 * MiB, de=True, byte_mode=True, name="stream_csv_128m_byte"),
        # bulk decoding, one wave of blocks and a little more
        _case("batch", "text", 256 * MiB, name="batch_text_2x256m"),
        # bulk decoding of records, several waves of blocks
        _case("batch", "csv", 512 * MiB, name="batch_csv_2x512m"),
        # a directory of uneven files in one launch
        _case("files", "mixed", 256 * MiB, name="files_256m"),
        # compressed data read from host memory for use on the GPU
        _case("from_host", "csv", 256 * MiB, de=True, name="from_host_csv_256m"),
        # host to host, as a drop-in for a host decompressor
        _case("host", "text", 128 * MiB, name="host_text_128m"),
        # writing streams: Huffman blocks of text, and byte-level blocks of records
        _case("compress", "text", 64 * MiB, name="compress_text_64m"),
        _case("compress", "csv", 16 * MiB + 4321, de=True, byte_mode=True, name="compress_csv_16m_byte"),
    ]


#: smallest and largest size of the drawn cases, by op
RANGES = {"stream": (4 * KiB, 256 * MiB), "batch": (1 * MiB, 256 * MiB), "files": (4 * MiB, 256 * MiB),
          "from_host": (1 * MiB, 256 * MiB), "host": (1 * MiB, 128 * MiB), "compress": (64 * KiB, 64 * MiB)}


def draw(rng: random.Random):
    op = rng.choice(["stream", "stream", "stream", "batch", "files", "from_host", "host", "compress"])
    lo, hi = RANGES[op]
    size = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return _case(op, "mixed" if op == "files" else rng.choice(["text", "csv"]), size, de=rng.random() < 0.5,
                 byte_mode=rng.random() < 0.25, block=rng.choice([64 * KiB, 100_000, 128 * KiB, 256 * KiB]),
                 n_sub=rng.choice([16, 32, 33, 64]), window=rng.choice([8 * KiB, 20_000, 32 * KiB]))


# ---------------------------------------------------------------------------
# inputs

_LETTERS = "etaoinshrdlcumwfgypbvkjxqz"
_PERCENT = [12.7, 9.1, 8.2, 7.5, 7.0, 6.7, 6.3, 6.1, 6.0, 4.3, 4.0, 2.8, 2.8, 2.4, 2.4, 2.2, 2.0, 2.0, 1.9, 1.5, 1.0,
            0.8, 0.15, 0.15, 0.1, 0.07]


def _quantised(weights):
    """4096-entry inverse distribution function of `weights`."""
    cdf = np.cumsum(np.asarray(weights, np.float64))
    return np.searchsorted(cdf / cdf[-1], (np.arange(4096) + 0.5) / 4096)


def _text(n, seed, dev):
    """n bytes of order-3 Markov text: the next byte is one of up to six
    successors of its context (weights 0.15^i) nine times in ten, else a letter
    by its frequency; in runs of 512 bytes made side by side."""
    w = np.full(256, 0.015 / 256)
    for ch, p in ((" ", 0.18), (".", 0.01), (",", 0.01), ("\n", 0.005)):
        w[ord(ch)] += p
    for ch, p in zip(_LETTERS, _PERCENT):
        w[ord(ch)] += 0.78 * p / sum(_PERCENT) * 0.96
        w[ord(ch.upper())] += 0.78 * p / sum(_PERCENT) * 0.04
    unigram = torch.from_numpy(_quantised(w)).to(dev)
    rank = torch.from_numpy(_quantised([0.9 * 0.85 * 0.15 ** i for i in range(6)] + [0.1])).to(dev)
    g = torch.Generator(device=dev).manual_seed(seed)
    run, chains = 512, -(-n // 512)
    out = torch.empty((run, chains), dtype=torch.uint8, device=dev)
    ctx = torch.randint(0, 64, (chains,), generator=g, device=dev)
    salt = (seed * 0x9E3779B97F4A7C1 + 0x632BE59B) % (1 << 62)
    for i in range(run):
        if i % 16 == 0:
            rnd = torch.randint(0, 1 << 24, (16, chains), generator=g, device=dev)
        r = rnd[i % 16]
        k = rank[r & 4095]
        h = (ctx * 0x2545F4914F6CDD1D + salt) * (2 * k + 1)
        h = (h ^ (h >> 29)) * 0x1B873593CC9E2D51
        b = unigram[torch.where(k == 6, r >> 12, (h >> 40) & 4095)]
        out[i] = b
        ctx = ((ctx << 8) | b) & 0xFFFFFF
    return out.t().reshape(-1)[:n].contiguous()


def _csv(n, seed, dev):
    """n bytes of rows of two ids (Zipf 1.1), two prices, two dates and two
    categories; one row in ten repeats one of the 64 before it but for a field."""
    g = torch.Generator(device=dev).manual_seed(seed)
    rows = n // 46 + 1  # no row is shorter
    py = random.Random(seed)

    def below(m, *shape):
        return torch.randint(0, m, shape or (rows,), generator=g, device=dev)

    def zipf(m):
        cdf = torch.cumsum(torch.arange(1, m + 1, device=dev, dtype=torch.float64) ** -1.1, 0)
        u = torch.rand(rows, generator=g, device=dev, dtype=torch.float64)
        return torch.searchsorted(cdf, u * cdf[-1]).clamp_(max=m - 1)

    cols = [zipf(999_999) + 1, zipf(999_999) + 1, below(999_999) + 1, below(999_999) + 1, below(1826), below(1826),
            zipf(20), zipf(20)]
    same, back, changed = below(10) == 0, below(64) + 1, below(8)
    src = (torch.arange(rows, device=dev) - back).clamp_(min=0)
    cols = [torch.where(same & (changed != f), c[src], c) for f, c in enumerate(cols)]
    parts, masks = [], []

    def digits(v, most, least=1):
        for k in range(most - 1, -1, -1):
            parts.append((v // 10 ** k % 10 + 48).to(torch.uint8)[:, None])
            masks.append(((v >= 10 ** k) | (k < least))[:, None])

    def table(strings, v):
        wide = max(map(len, strings))
        t = np.zeros((len(strings), wide), np.uint8)
        for i, s in enumerate(strings):
            t[i, :len(s)] = np.frombuffer(s.encode(), np.uint8)
        parts.append(torch.from_numpy(t).to(dev)[v])
        masks.append(parts[-1] != 0)

    def mark(ch):
        parts.append(torch.full((rows, 1), ord(ch), dtype=torch.uint8, device=dev))
        masks.append(torch.ones((rows, 1), dtype=torch.bool, device=dev))

    day0 = datetime.date(2015, 1, 1)
    days = [(day0 + datetime.timedelta(d)).isoformat() for d in range(1826)]
    tokens = ["".join(py.choice(_LETTERS) for _ in range(py.randint(4, 12))) for _ in range(20)]
    for f, c in enumerate(cols):
        if f < 2:
            digits(c, 6)
        elif f < 4:
            digits(c // 100, 4)
            mark(".")
            digits(c % 100, 2, 2)
        else:
            table(days if f < 6 else tokens, c)
        mark("," if f < 7 else "\n")
    return torch.cat(parts, 1)[torch.cat(masks, 1)][:n].contiguous()


def _data(kind, n, seed):
    return (_text if kind == "text" else _csv)(n, seed, torch.device("cuda")).cpu().numpy()


def _compress(case, data, de):
    return gmp.compress(data, case["block"], case["n_sub"], case["window"], de=de, byte_mode=case["byte_mode"])


def _pinned(n):
    return torch.empty(n, dtype=torch.uint8, pin_memory=True).numpy()


def _files(case):
    """(kind, de, bytes) of files whose sizes add up to the case's."""
    rng, left, files = random.Random(case["bytes"]), case["bytes"], []
    while left:
        size = min(left, int(math.exp(rng.uniform(math.log(FILE_MIN), math.log(FILE_MAX)))))
        files.append((rng.choice(["text", "csv"]), rng.random() < 0.5, size))
        left -= size
    return files


def prepare(case, seed):
    op, n = case["op"], case["bytes"]
    if op == "compress":
        # `kept`: where the program collects its streams (here the latest, then zeros)
        return {"case": case, "data": _data(case["data"], n, seed), "kept": np.zeros(n + n // 4 + 64 * KiB, np.uint8),
                "size": 0}
    state = {"case": case, "ctx": gmp.Context(max_block_out=case["block"])}
    if op in ("from_host", "host"):
        stream = _compress(case, _data(case["data"], n, seed), case["de"])
        state["stream"] = _pinned(stream.size)
        state["stream"][:] = stream
        state["out"] = _pinned(n) if op == "host" else torch.zeros(n, dtype=torch.uint8, device="cuda")
        return state
    if op == "files":
        files, streams, sizes = _files(case), [], []
        pool = {k: _data(k, max(sum(s for kind, _, s in files if kind == k), 1), seed) for k in ("text", "csv")}
        used = {"text": 0, "csv": 0}
        for kind, de, size in files:
            streams.append(_compress(case, pool[kind][used[kind]:used[kind] + size], de))
            used[kind] += size
            sizes.append(size)
    else:
        data = _data(case["data"], n, seed)
        streams = [_compress(case, data, de) for de in ([False, True] if op == "batch" else [case["de"]])]
        sizes = [n] * len(streams)
    state["streams"] = [gmp.DeviceStream(s) for s in streams]
    starts = np.concatenate([[0], np.cumsum([-(-s // 256) * 256 for s in sizes])])
    state["out"] = torch.zeros(int(starts[-1]), dtype=torch.uint8, device="cuda")
    state["status"] = torch.zeros(len(streams), dtype=torch.int32, device="cuda")
    if op != "stream":
        state["table"] = gmp.make_file_table([d.file_desc(state["out"][a:a + s])
                                              for d, a, s in zip(state["streams"], starts.tolist(), sizes)])
    if op == "files":
        state["graph"] = state["ctx"].batch_graph(state["table"], len(streams), state["status"])
    return state


def run(state):
    case, ctx = state["case"], state.get("ctx")
    op = case["op"]
    if op == "compress":
        stream = gmp.compress_gpu(state["data"], case["block"], case["n_sub"], case["window"], de=case["de"],
                                  byte_mode=case["byte_mode"])
        kept, before, state["size"] = state["kept"], state["size"], stream.size
        kept[:stream.size] = stream
        kept[stream.size:before] = 0
        return stream.size, kept
    if op == "host":
        return ctx.decompress_host_batch([state["stream"]], [state["out"]])
    if op == "from_host":
        return ctx.decompress_from_host_batch([state["stream"]], [state["out"]])
    if op == "stream":
        ctx.decompress_into(state["streams"][0], state["out"], state["status"])
    elif op == "batch":
        ctx.decompress_batch(state["table"], len(state["streams"]), state["status"])
    else:
        state["graph"].launch()
    return state["out"], state["status"]


def work(case):
    """Decompressed bytes once and compressed bytes (at the kind's usual ratio)
    once; no floating-point work."""
    ratio = {"text": 2.7, "csv": 3.0, "mixed": 2.85}[case["data"]] * (0.64 if case["byte_mode"] else 1.0)
    return {"bytes": (2 if case["op"] == "batch" else 1) * case["bytes"] * (1 + 1 / ratio), "flops": 0}

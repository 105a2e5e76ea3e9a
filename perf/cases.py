"""Timed cases of the decode path: what programs that train from PCR records call, over the range of records they hold.

A case names an operation, a kind of record and a fidelity:

  op        decode   pcr_decode of a record whose handle is kept (an epoch over records held in device memory)
            raise    pcr_decode at k0, then pcr_decode_more to k (fidelity switched while training)
            tensor   pcr_decode_tensor: random-resized crops, flips, normalisation, straight to a training batch
            loader   a record that arrives in pinned host memory: open, decode, wait, read the status, close
  shape     tiny32, imagenet, celeba, ham: image sizes and content of the benchmark's workloads; mixed: sides from 33 to
            640 pixels, mostly odd
  n         images of the record
  restart   restart markers once per MCU row (True) or none (False)
  script    ten: the ten-scan progressive script; baseline: one sequential scan
  sampling  chroma sampling: 420, 422, 440, 444, grey
  upsample  replicate or triangle (4:2:0, op decode)
  k, k0     scan groups decoded
  size, dtype  of the training batch

Records are made from the seed by the repository's generator: at most about ten million pixels of distinct images, which
larger records repeat (every copy has bytes, coefficients and pixels of its own).
"""
from __future__ import annotations

import functools
import math
import random
import struct

import numpy as np
import torch

import pcr_synth
from paper_1911_00472_b200 import Decoder

MEAN, STD = (0.485, 0.456, 0.406), (0.229, 0.224, 0.225)
DTYPES = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
SAMPLINGS = {"420": (2, 2, 3), "422": (2, 1, 3), "440": (1, 2, 3), "444": (1, 1, 3), "grey": (1, 1, 1)}
WORKLOAD = {"tiny32": 0, "imagenet": 1, "celeba": 2, "ham": 3, "mixed": 1}
DISTINCT_PIXELS = 10_000_000


def _case(name, op, shape, n, k, **more):
    c = {"name": name, "op": op, "shape": shape, "n": n, "k": k, "k0": 0, "restart": True, "script": "ten", "sampling": "420",
         "upsample": "replicate", "size": 0, "dtype": "none"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest record: nothing but launches and waits
        _case("tiny32_32_k10", "decode", "tiny32", 32, 10),
        # the benchmark's record at the fidelities the paper trains at
        _case("imagenet_1024_k1", "decode", "imagenet", 1024, 1),
        _case("imagenet_1024_k5", "decode", "imagenet", 1024, 5),
        _case("imagenet_1024_k10", "decode", "imagenet", 1024, 10),
        # rows that start at any byte address, images that end inside an MCU
        _case("celeba_1024_k10", "decode", "celeba", 1024, 10),
        # large images without restart markers; the largest case
        _case("ham_1024_k10", "decode", "ham", 1024, 10, restart=False),
        # the same at the paper's middle fidelity, a record of ordinary size
        _case("ham_256_k5", "decode", "ham", 256, 5, restart=False),
        # conventional JPEGs, the paper's comparison
        _case("imagenet_1024_baseline", "decode", "imagenet", 1024, 1, script="baseline"),
        # images of all sizes without chroma subsampling
        _case("mixed_96_444_k10", "decode", "mixed", 96, 10, sampling="444"),
        # a training batch, the usual augmentation
        _case("imagenet_1024_tensor_k5", "tensor", "imagenet", 1024, 5, size=224, dtype="f16"),
        # fidelity raised while training
        _case("imagenet_512_raise_2_10", "raise", "imagenet", 512, 10, k0=2),
        # records streamed from host memory, each seen once
        _case("imagenet_1024_loader_k10", "loader", "imagenet", 1024, 10),
    ]


def draw(rng: random.Random):
    shape = rng.choice(["tiny32", "imagenet", "imagenet", "imagenet", "celeba", "ham", "mixed", "mixed"])
    op = rng.choice(["decode", "decode", "decode", "raise", "tensor", "loader"])
    sampling = rng.choice(["420", "420", "420", "422", "440", "444", "grey"])
    most = 512 if shape == "ham" or sampling == "444" else 1024
    n = int(round(math.exp(rng.uniform(math.log(4), math.log(most)))))
    script = "baseline" if op != "raise" and rng.random() < 0.15 else "ten"
    groups = 1 if script == "baseline" else (6 if sampling == "grey" else 10)
    k = rng.randint(2 if op == "raise" else 1, groups)
    c = _case("", op, shape, n, k, script=script, sampling=sampling, restart=rng.random() < (0.3 if shape == "ham" else 0.7))
    del c["name"]
    if op == "raise":
        c["k0"] = rng.randint(1, k - 1)
    if op == "decode" and sampling == "420" and rng.random() < 0.25:
        c["upsample"] = "triangle"
    if op == "tensor":
        c["size"], c["dtype"] = rng.choice([160, 224]), rng.choice(["f16", "bf16", "f32"])
    return c


def _specs(case, seed):
    """Per-image recipes of the record's distinct images."""
    w = pcr_synth.WORKLOADS[WORKLOAD[case["shape"]]]
    sizes = random.Random(case["n"])              # sizes belong to the case, contents to the seed
    rng = random.Random(seed)
    specs, pixels = [], 0
    while len(specs) < case["n"] and pixels < DISTINCT_PIXELS:
        if case["shape"] == "mixed":
            W, H = (int(round(math.exp(sizes.uniform(math.log(33), math.log(640))))) for _ in range(2))
        elif w.fixed_size is not None:
            W, H = w.fixed_size
        else:
            W, H = (16 * int(round(sizes.uniform(256, 500) / 16.0)) for _ in range(2))
        specs.append(pcr_synth.ImageSpec(W, H, rng.randrange(1000), w.quality, w.beta, w.gamma, w.sigma, 1 if w.blobs else 0, 0,
                                         rng.getrandbits(62)))
        pixels += W * H
    return specs


def _repeat(rec: np.ndarray, n: int) -> np.ndarray:
    """The record of n images that repeats the images of `rec` in order."""
    N, G = struct.unpack_from("<II", rec, 8)
    meta_off, index_off = struct.unpack_from("<QQ", rec, 24)
    meta = rec[meta_off:meta_off + 16 * N].reshape(N, 16)
    ends = rec[index_off:index_off + 8 * (G + 1)].view(np.uint64).astype(np.int64)
    at = index_off + 8 * (G + 1)
    chunks = np.frombuffer(rec[at:at + 16 * G * N].tobytes(), dtype=[("off", "<u8"), ("len", "<u4"), ("rsvd", "<u4")]).reshape(G, N)
    rounds, rest = divmod(n, N)
    idx = np.arange(n) % N
    new_meta = 64
    new_index = new_meta + 16 * n
    pos = (new_index + 8 * (G + 1) + 16 * G * n + 15) // 16 * 16
    new_ends, new_chunks, parts = [pos], np.zeros((G, n), chunks.dtype), []
    for g in range(G):
        begin, size = int(ends[g]), int(ends[g + 1] - ends[g])
        part = size if rest == 0 else int(chunks["off"][g, rest]) - begin       # chunks lie in image order
        data = rec[begin:begin + size]
        parts += [data] * rounds + ([data[:part]] if rest else [])
        new_chunks["off"][g] = chunks["off"][g, idx].astype(np.int64) - begin + pos + np.arange(n) // N * size
        new_chunks["len"][g] = chunks["len"][g, idx]
        pos += rounds * size + (part if rest else 0)
        new_ends.append(pos)
    out = np.zeros(pos, dtype=np.uint8)
    out[:64] = rec[:64]
    struct.pack_into("<I", out, 8, n)
    struct.pack_into("<QQQQ", out, 24, new_meta, new_index, new_ends[0], pos)
    out[new_meta:new_meta + 16 * n] = meta[idx].reshape(-1)
    out[new_index:new_index + 8 * (G + 1)] = np.array(new_ends, dtype=np.uint64).view(np.uint8)
    out[new_index + 8 * (G + 1):new_index + 8 * (G + 1) + 16 * G * n] = np.frombuffer(new_chunks.tobytes(), dtype=np.uint8)
    out[new_ends[0]:] = np.concatenate(parts)
    return out


def _record(case, seed):
    """(record bytes, (width, height) of every image)"""
    specs = _specs(case, seed)
    with pcr_synth.sampling(*SAMPLINGS[case["sampling"]]):
        with pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE if case["script"] == "baseline" else pcr_synth.SCRIPT_DEFAULT):
            rec = pcr_synth.record_from_specs(specs, restart_rows=case["restart"])
    raw, dims = rec.bytes, rec.dims
    rec.close()
    n = case["n"]
    return (raw if n == len(dims) else _repeat(raw, n)), [dims[i % len(dims)] for i in range(n)]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    raw, s.dims = _record(case, seed)
    s.raw = torch.from_numpy(raw).pin_memory().numpy()       # the loader's read buffer
    dec = Decoder(s.raw, device="cuda:0")
    s.out = torch.zeros(dec.out_bytes, dtype=torch.uint8, device="cuda:0")
    s.dec = dec
    if case["op"] == "loader":
        dec.close()
        s.dec = None
    if case["op"] == "raise":
        s.first = torch.zeros_like(s.out)
    if case["op"] == "tensor":
        s.crops = pcr_synth.random_resized_crops(s.dims, seed=seed)
        s.tensor = torch.zeros((case["n"], 3, case["size"], case["size"]), dtype=DTYPES[case["dtype"]], device="cuda:0")
    if case["upsample"] == "triangle":
        dec.set_upsampling(True)
    return s


def run(s):
    op, k = s.case["op"], s.case["k"]
    if op == "decode":
        return {"rgb": s.dec.decode(k, s.out)}
    if op == "raise":
        first = s.dec.decode(s.case["k0"], s.first)
        return {"first": first, "rgb": s.dec.decode_more(k, s.out)}
    if op == "tensor":
        return {"batch": s.dec.decode_tensor(k, s.crops, s.case["size"], MEAN, STD, DTYPES[s.case["dtype"]], rgb=s.out, tensor=s.tensor)}
    dec = Decoder(s.raw, device="cuda:0")
    dec.decode(k, s.out)
    torch.cuda.current_stream().synchronize()
    bad, code = dec.status()
    dec.close()
    return {"rgb": s.out, "bad": bad, "code": code}


@functools.lru_cache(maxsize=None)
def _prefix_bytes(key, k):
    raw, dims = _record(dict(key), 0)
    index_off = struct.unpack_from("<Q", raw, 32)[0]
    return struct.unpack_from("<Q", raw, index_off + 8 * k)[0], tuple(dims)


def work(case):
    """Bytes: the record up to scan group k read once, the pixels (or the batch) written once.  Operations: integer
    operations of dequantisation, inverse transform (16 eight-point transforms of about 50 operations a block) and colour."""
    key = tuple(sorted((a, b) for a, b in case.items() if a in ("shape", "n", "restart", "script", "sampling")))
    prefix, dims = _prefix_bytes(key, case["k"])
    hs, vs, nc = SAMPLINGS[case["sampling"]]
    if case["op"] == "tensor":
        crops = pcr_synth.random_resized_crops(dims, seed=0)
        pixels = float(np.sum(crops[:, 2].astype(np.float64) * crops[:, 3]))
        values = 3.0 * case["n"] * case["size"] ** 2
        written, extra = values * (4 if case["dtype"] == "f32" else 2), 12.0 * values
    else:
        pixels = float(sum(W * H for W, H in dims))
        written, extra = 3.0 * pixels, 0.0
    passes = 2 if case["op"] == "raise" else 1
    samples = pixels * (1.0 + (2.0 / (hs * vs) if nc == 3 else 0.0))
    return {"bytes": prefix + passes * written, "flops": passes * (13.5 * samples + 10.0 * pixels) + extra}


def tolerance(case):
    if case["op"] != "tensor":
        return "exact"
    # single-precision interpolation and one rounding to the output type
    return {"f16": {"rel": 5e-4, "max": 2e-3}, "bf16": {"rel": 4e-3, "max": 1.6e-2}, "f32": {"rel": 2e-6, "max": 2e-5}}[case["dtype"]]

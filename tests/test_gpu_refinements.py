"""AC refinements of scans with restart intervals, by the CTAs that take them in small launches and by the lane-per-interval
warps of large ones (PCR_REFINE_CTAS, read when a record is opened, chooses), in pairs of scans and one after the other
(PCR_PAIRS): intervals of one block to several rows, runs of blocks that last a whole interval, blocks as long as the format allows, streams that are cut short."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from oracle import pcr_oracle as O
from test_gpu_kernel_edges import _compare, _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("ctas", [0, 1 << 20])
@pytest.mark.parametrize("fixed", [0, 1, 7, 150])
@pytest.mark.parametrize("kind", ["dense", "wide", "sparse", "empty"])
def test_blocks_and_intervals(kind, fixed, ctas, pairs, monkeypatch):
    """fixed: MCUs an interval (0: a row).  dense: every block takes nearly as many bits as one can; wide: rows of 90 blocks,
    a few rounds of lists; sparse and empty: end-of-band runs over blocks, rows and whole intervals."""
    rng = np.random.default_rng(fixed)
    dims = [(90, 41), (8, 8), (33, 70)] if kind != "wide" else [(720, 24), (200, 40)]
    density = {"dense": 1.0, "wide": 0.3, "sparse": 0.004, "empty": 0.0}[kind]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), density, 1023 if kind == "dense" else 20) for w, h in dims]
    rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=fixed == 0, restart_fixed=fixed)
    monkeypatch.setenv("PCR_REFINE_CTAS", str(ctas))
    monkeypatch.setenv("PCR_PAIRS", str(pairs))
    _compare(rec, (6, 9, 10))


@pytest.mark.parametrize("restart_rows", [True, False])
def test_corrections_by_halves(restart_rows, monkeypatch):
    """Correction bits of the pixel stage: blocks whose earlier coefficients fill one half of the positions, both or none, with the last
    set bit in either half, at its end, or nowhere, and new coefficients among them."""
    rng = np.random.default_rng(11)
    dims = [(200, 120), (8, 8), (90, 41)]
    coeffs = []
    for w, h in dims:
        nb = pcr_synth.num_blocks(w, h)
        c = np.zeros((nb, 64), dtype=np.int16)
        first, second = rng.choice([0.0, 0.1, 1.0], size=nb), rng.choice([0.0, 0.1, 1.0], size=nb)
        for lo, hi, share in ((1, 32, first), (32, 64, second)):
            # (4: earlier than every refinement; two low bits: none set, one, or any)
            low = rng.integers(0, 4, size=(nb, hi - lo)) * (rng.random((nb, hi - lo)) < rng.choice([0.0, 0.03, 1.0], size=nb)[:, None])
            low[rng.random(nb) < 0.1, -1] = 3
            old = rng.random((nb, hi - lo)) < share[:, None]
            new = ~old & (rng.random((nb, hi - lo)) < rng.choice([0.0, 0.05], size=nb)[:, None])
            c[:, lo:hi] = (old * (4 + low) + new * rng.integers(1, 4, size=(nb, hi - lo))) * rng.choice([-1, 1], size=(nb, hi - lo))
        c[:, 0] = rng.integers(-500, 501, nb)
        coeffs.append(c)
    monkeypatch.setenv("PCR_LONG_MIN_BYTES", "0")
    _compare(pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=restart_rows), (6, 9, 10))


@pytest.mark.parametrize("scan", [5, 9])
@pytest.mark.parametrize("ctas", [0, 1 << 20])
def test_damaged_interval(ctas, scan, monkeypatch):
    """The second half of one restart interval of one image replaced by ones (no code is all ones): that image is reported,
    the others' pixels are the oracle's."""
    import struct
    import torch
    from paper_1911_00472_b200 import Decoder
    rng = np.random.default_rng(scan)
    dims = [(120, 60), (90, 41), (33, 70)]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), 0.3, 20) for w, h in dims]
    rec = pcr_synth.record_from_coeffs(dims, coeffs)
    bad = np.array(rec.bytes, copy=True)
    n, groups = struct.unpack_from("<II", bad, 8)
    index = struct.unpack_from("<Q", bad, 32)[0] + 8 * (groups + 1)
    off, length = struct.unpack_from("<QI", bad, index + 16 * (scan * n + 1))
    chunk = bad[off:off + length].tobytes()
    head = chunk.index(b"\xff\xda")
    data = head + 2 + struct.unpack_from(">H", chunk, head + 2)[0]
    first, end = chunk.index(b"\xff\xd0", data) + 2, chunk.index(b"\xff\xd1", data)       # the second interval
    begin = (first + end) // 2
    begin += (end - begin) % 2
    assert end - begin >= 8
    bad[off + begin:off + end] = np.tile(np.array([0xFF, 0], dtype=np.uint8), (end - begin) // 2)
    monkeypatch.setenv("PCR_REFINE_CTAS", str(ctas))
    dec = Decoder(bad)
    try:
        out = dec.decode(10)
        torch.cuda.synchronize()
        assert dec.status() == (1, -3)
        pixels = out.cpu().numpy()
        for i in (0, 2):
            want = O.decode_image(rec.bytes, i, 10)[1]
            inf = dec.info[i]
            assert np.array_equal(pixels[inf.out_offset:inf.out_offset + inf.out_bytes].reshape(want.shape), want), i
    finally:
        dec.close()

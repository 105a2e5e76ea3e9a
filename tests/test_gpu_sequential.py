"""Baseline records with restart intervals, by CTAs that follow 32 intervals' symbols while other warps write the blocks and by the
lane-per-interval warps of large launches (PCR_SEQ_CTAS, read when a record is opened, chooses): intervals of one MCU to several
rows, blocks as long as the format allows and of two symbols, every chroma sampling (the blocks of an MCU change tables in
different places), an interval that is damaged."""
from __future__ import annotations

import struct

import numpy as np
import pytest

import helpers
import pcr_synth
from oracle import pcr_oracle as O
from test_gpu_kernel_edges import _compare, _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [0, 1 << 20])
@pytest.mark.parametrize("samp", [(2, 2, 3), (2, 1, 3), (1, 2, 3), (1, 1, 3), (1, 1, 1)])
@pytest.mark.parametrize("fixed", [0, 1, 5, 60])
@pytest.mark.parametrize("kind", ["dense", "usual", "empty"])
def test_blocks_and_intervals(kind, fixed, samp, ctas, monkeypatch):
    """fixed: MCUs an interval (0: a row).  dense: blocks of up to 64 symbols of many bits; empty: two symbols a block, so that a
    round ends most blocks there can be."""
    rng = np.random.default_rng(fixed)
    dims = [(330, 33), (8, 8), (90, 41)]
    density, top = {"dense": (1.0, 1023), "usual": (0.15, 40), "empty": (0.0, 1)}[kind]
    with pcr_synth.sampling(*samp), pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), density, top) for w, h in dims]
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=fixed == 0, restart_fixed=fixed)
    monkeypatch.setenv("PCR_SEQ_CTAS", str(ctas))
    _compare(rec, (1,))


@pytest.mark.parametrize("samp", [(2, 2, 3), (1, 2, 3), (1, 1, 1)])
def test_flat_rows(samp):
    """Blocks of two symbols, hundreds of them an interval: round after round ends as many blocks as it can.  (The DC differences go
    up and down, so a block read from another one's beginning shows.)"""
    rng = np.random.default_rng(3)
    dims = [(1600, 24), (800, 48), (130, 17)]
    with pcr_synth.sampling(*samp), pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), 0.0, 40) for w, h in dims]
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=True)
    _compare(rec, (1,))


@pytest.mark.parametrize("ctas", [0, 1 << 20])
def test_damaged_interval(ctas, monkeypatch):
    """The second half of one restart interval of one image replaced by ones (no code is all ones): that image is reported,
    the others' pixels are the oracle's."""
    import torch
    from paper_1911_00472_b200 import Decoder
    rng = np.random.default_rng(1)
    dims = [(120, 60), (90, 41), (33, 70)]
    with pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE):
        rec = pcr_synth.record_from_coeffs(dims, [_field(rng, pcr_synth.num_blocks(w, h), 0.3, 20) for w, h in dims])
    bad = np.array(rec.bytes, copy=True)
    n, groups = struct.unpack_from("<II", bad, 8)
    index = struct.unpack_from("<Q", bad, 32)[0] + 8 * (groups + 1)
    off, length = struct.unpack_from("<QI", bad, index + 16)
    chunk = bad[off:off + length].tobytes()
    head = chunk.index(b"\xff\xda")
    data = head + 2 + struct.unpack_from(">H", chunk, head + 2)[0]
    first, end = chunk.index(b"\xff\xd0", data) + 2, chunk.index(b"\xff\xd1", data)
    begin = (first + end) // 2
    begin += (end - begin) % 2
    bad[off + begin:off + end] = np.tile(np.array([0xFF, 0], dtype=np.uint8), (end - begin) // 2)
    monkeypatch.setenv("PCR_SEQ_CTAS", str(ctas))
    dec = Decoder(bad)
    try:
        out = dec.decode(1)
        torch.cuda.synchronize()
        assert dec.status() == (1, -3)
        pixels = out.cpu().numpy()
        for i in (0, 2):
            want = O.decode_image(rec.bytes, i, 1)[1]
            inf = dec.info[i]
            assert np.array_equal(pixels[inf.out_offset:inf.out_offset + inf.out_bytes].reshape(want.shape), want), i
    finally:
        dec.close()


@pytest.mark.parametrize("form", ["ctas", "lanes", "no markers"])
@pytest.mark.parametrize("block", [0, 3])
def test_coefficient_behind_the_block(block, form, monkeypatch):
    """A run of fifteen zeros instead of fourteen puts a block's last coefficient at position 64: the image is reported, the blocks
    behind it keep their places, and the other images are untouched."""
    dims = [(64, 24), (72, 24), (24, 64)]
    with pcr_synth.sampling(1, 1, 1), pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE), pcr_synth.ac_code_length(10):
        coeffs = [np.zeros((pcr_synth.num_blocks(w, h), 64), dtype=np.int16) for w, h in dims]
        for c in coeffs:
            c[:, 63] = 1                                       # three runs of sixteen zeros, fourteen zeros and the one
            c[-1, 16] = 1                                      # (gives the longer run a code)
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=form != "no markers")
    bad = np.array(rec.bytes, copy=True)
    begin, end, tables = helpers.entropy_data(bad, 1, 0)
    codes = tables[0]
    (zeros, n), (short, m), (long, l) = codes[0xF0], codes[0xE1], codes[0xF1]
    assert m == l
    text = "".join(f"{b:08b}" for b in bytes(bad[begin:end]).replace(b"\xff\0", b"\xff"))
    block_text = 3 * f"{zeros:0{n}b}" + f"{short:0{m}b}"
    at = -1
    for _ in range(block + 1):
        at = text.index(block_text, at + 1)
    if form != "no markers":
        end = begin + bytes(bad[begin:end]).index(b"\xff\xd0")
    helpers.overwrite_bits(bad, begin, end, at + 3 * n, f"{long:0{l}b}")
    monkeypatch.setenv("PCR_SEQ_CTAS", "0" if form == "lanes" else str(1 << 20))
    monkeypatch.setenv("PCR_LONG_MIN_BYTES", "0")
    helpers.decode_damaged(bad, rec.bytes, 1, 1)

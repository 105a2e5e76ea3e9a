"""The kernels' forms for small and for large launches, forced on small records (the PCR_* variables are read when a record is
opened): raising the fidelity of a resident decode, training batches that decode only the rows their crops touch, and
randomised records with the forms drawn too.  Everything against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from oracle import pcr_oracle as O
from test_gpu_kernel_edges import _field
from test_gpu_random_records import _one
from test_gpu_tensor import _check

pytestmark = pytest.mark.gpu

MANY = str(1 << 20)
FORMS = {
    "small": dict(PCR_REFINE_CTAS=MANY, PCR_PAIRS="1", PCR_PACK_WARPS=MANY, PCR_SHORT_WARPS=MANY, PCR_INDEX_CTAS=MANY, PCR_LONG_CTAS=MANY, PCR_SEQ_CTAS=MANY),
    "large": dict(PCR_REFINE_CTAS="0", PCR_PAIRS="0", PCR_PACK_WARPS="0", PCR_SHORT_WARPS=MANY, PCR_INDEX_CTAS="0", PCR_LONG_CTAS="0", PCR_SEQ_CTAS="0"),
    "pairs of lanes, short intervals": dict(PCR_REFINE_CTAS="0", PCR_PAIRS="1", PCR_PACK_WARPS=MANY, PCR_SHORT_WARPS="0", PCR_INDEX_CTAS="0"),
    "CTAs without pairs, slices": dict(PCR_REFINE_CTAS=MANY, PCR_PAIRS="0", PCR_PACK_WARPS="0", PCR_SLICES="3"),
}


def _set(form, monkeypatch):
    for name, value in FORMS[form].items():
        monkeypatch.setenv(name, value)


def _record(restart, script=None, samp=(2, 2, 3)):
    rng = np.random.default_rng(5)
    dims = [(200, 90), (33, 150), (90, 41), (8, 8), (320, 200)]
    with pcr_synth.scan_script(script), pcr_synth.sampling(*samp):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), d, 40) for (w, h), d in zip(dims, (0.15, 0.5, 0.02, 1.0, 0.1))]
        return pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=restart)


@pytest.mark.parametrize("restart", [True, False])
@pytest.mark.parametrize("form", list(FORMS))
def test_raised_fidelity(form, restart, monkeypatch):
    import torch
    from paper_1911_00472_b200 import Decoder, pcr_image_blocks
    rec = _record(restart)
    _set(form, monkeypatch)
    dec = Decoder(rec.bytes)
    try:
        for chain in ([1, 10], [2, 6, 10], [5, 10], [6, 9, 10], [3, 7, 8]):
            for k in chain:
                out = dec.decode(k) if k == chain[0] else dec.decode_more(k)
            torch.cuda.synchronize()
            assert dec.status() == (-1, 0), chain
            pixels, coeffs = out.cpu().numpy(), dec.coeffs().cpu().numpy()
            for i in range(rec.n_images):
                want_c, want = O.decode_image(rec.bytes, i, chain[-1])
                inf = dec.info[i]
                a, b = pcr_image_blocks(dec.handle, i)
                assert np.array_equal(coeffs[a:a + b], want_c), (chain, i)
                assert np.array_equal(pixels[inf.out_offset:inf.out_offset + inf.out_bytes].reshape(want.shape), want), (chain, i)
    finally:
        dec.close()


@pytest.mark.parametrize("script", ["ten", "baseline"])
@pytest.mark.parametrize("restart", [True, False])
@pytest.mark.parametrize("form", list(FORMS))
def test_crops(form, restart, script, monkeypatch):
    """Crops of a few rows in the middle, of one row and of whole images: intervals above and below are left out.  (Source coordinates up to
    320 are exact to 2^-16 of a pixel in single precision, neighbouring pixels differ by up to 255 / 255 / 0.224 = 4.5: 7e-5 before the
    result is rounded, below half a unit of half precision, so one unit as in test_gpu_tensor.)"""
    rec = _record(restart, pcr_synth.SCRIPT_BASELINE if script == "baseline" else None)
    crops = pcr_synth.random_resized_crops([(int(w), int(h)) for w, h in rec.dims], 3)
    crops[1] = (3, 70, 20, 9, 1)
    crops[2] = (0, 40, 90, 1, 0)
    crops[4] = (100, 101, 60, 33, 1)
    _set(form, monkeypatch)
    for k in ((1,) if script == "baseline" else (1, 5, 6, 10)):
        _check(rec, k, crops, 24, range(rec.n_images), "float16")


@pytest.mark.parametrize("first", [1000, 1040])
def test_random_records(first, monkeypatch):
    for seed in range(first, first + 40):
        rng = np.random.default_rng(seed + 7)
        for name in ("PCR_REFINE_CTAS", "PCR_PAIRS", "PCR_PACK_WARPS", "PCR_SHORT_WARPS", "PCR_INDEX_CTAS", "PCR_LONG_CTAS", "PCR_SEQ_CTAS"):
            monkeypatch.setenv(name, str(int(rng.choice([0, 1 << 20]))))
        _one(seed, monkeypatch)

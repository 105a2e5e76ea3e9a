"""First passes and sequential scans that are one restart interval, by narrow and by wide CTAs (PCR_LONG_CTAS, read when a record is
opened, chooses): fewer subsequences than threads and as many, every chroma sampling (the places of the MCU that a DC scan
is read from), single-component DC scans, one table for all components and tables that differ."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from test_gpu_kernel_edges import _compare, _field

pytestmark = pytest.mark.gpu

SINGLE = [((2,), 0, 0, 0, 0), ((0,), 0, 0, 0, 1), ((1,), 0, 0, 0, 0), ((0,), 1, 63, 0, 0), ((1,), 1, 7, 0, 0), ((2,), 8, 63, 0, 0)]


@pytest.mark.parametrize("ctas", [0, 1 << 20])
@pytest.mark.parametrize("samp", [(2, 2, 3), (2, 1, 3), (1, 2, 3), (1, 1, 3), (1, 1, 1)])
@pytest.mark.parametrize("script", ["ten", "baseline", "single"])
def test_subsequences(script, samp, ctas, monkeypatch):
    if script == "single" and samp[2] == 1:
        pytest.skip("a greyscale record has one component")
    rng = np.random.default_rng(samp[0] + 2 * samp[1] + 4 * samp[2])
    dims = [(40, 24), (330, 200), (500, 330), (104, 400)]
    chosen = {"ten": None, "baseline": pcr_synth.SCRIPT_BASELINE, "single": SINGLE}[script]
    with pcr_synth.sampling(*samp), pcr_synth.scan_script(chosen):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), float(rng.uniform(0.02, 0.4)), 60) for w, h in dims]
        # differences of one size almost everywhere: readings from a wrong place of the MCU go on unnoticed
        coeffs[2][:, 0] = np.cumsum(rng.integers(0, 2, len(coeffs[2]))) % 7
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=False)
    monkeypatch.setenv("PCR_LONG_MIN_BYTES", "0")
    monkeypatch.setenv("PCR_LONG_CTAS", str(ctas))
    last = {"ten": 6 if samp[2] == 1 else 10, "baseline": 1, "single": 6}[script]
    _compare(rec, sorted({1, min(5, last), last}))


@pytest.mark.parametrize("ctas", [0, 1 << 20])
@pytest.mark.parametrize("samp", [(2, 2, 3), (2, 1, 3), (1, 2, 3), (1, 1, 3)])
@pytest.mark.parametrize("length", [350, 1000])
def test_flat_stretches(length, samp, ctas, monkeypatch):
    """DC scans with long stretches of one code: readings that begin inside one fall in late or not at all, so that some subsequences
    have to be read once more, some behind others."""
    rng = np.random.default_rng(length // 50)
    dims = [(640, 400), (400, 640), (96, 1000)]
    with pcr_synth.sampling(*samp):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), 0.0, 1) for w, h in dims]
        for c in coeffs:
            c[np.repeat(rng.random(len(c) // length + 1) < 0.6, length)[:len(c)], 0] = 7
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=False)
    monkeypatch.setenv("PCR_LONG_CTAS", str(ctas))
    _compare(rec, (1,))

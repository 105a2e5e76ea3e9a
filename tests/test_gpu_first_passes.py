"""First passes in scans with restart intervals, with their stores packed (much data) and one by one (PCR_PACK_WARPS, read when a
record is opened, chooses), and in the form for many short intervals (PCR_SHORT_WARPS): bands that hold whole words of a block's
positions 1..7, parts of words or none, intervals of one block to several rows, lists of values that end anywhere in a group
of four, codes longer than the tables' index."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from test_gpu_kernel_edges import _compare, _field

pytestmark = pytest.mark.gpu

SCRIPTS = {
    "ten": None,
    "odd": [((0, 1, 2), 0, 0, 0, 0), ((0,), 1, 3, 0, 0), ((0,), 4, 4, 0, 0), ((0,), 5, 9, 0, 1), ((0,), 10, 63, 0, 0), ((1,), 1, 2, 0, 0),
            ((1,), 3, 63, 0, 0), ((2,), 2, 63, 0, 0), ((2,), 1, 1, 0, 0)],
    "single": [((2,), 0, 0, 0, 0), ((0,), 0, 0, 0, 1), ((1,), 0, 0, 0, 0), ((0,), 1, 63, 0, 0), ((1,), 1, 7, 0, 0), ((2,), 8, 63, 0, 0)],
}


@pytest.mark.parametrize("warps", [0, 1 << 20])
@pytest.mark.parametrize("fixed", [0, 1, 7])
@pytest.mark.parametrize("script", list(SCRIPTS))
def test_bands_and_intervals(script, fixed, warps, monkeypatch):
    rng = np.random.default_rng(fixed)
    dims = [(200, 33), (8, 8), (90, 41)]
    with pcr_synth.scan_script(SCRIPTS[script]):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), d, t) for (w, h), d, t in zip(dims, (0.15, 1.0, 0.02), (60, 1023, 500))]
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=fixed == 0, restart_fixed=fixed)
    monkeypatch.setenv("PCR_PACK_WARPS", str(warps))
    _compare(rec, (1, 5) if script == "ten" else range(1, len(SCRIPTS[script]) + 1))


@pytest.mark.parametrize("fixed", [0, 1, 7])
@pytest.mark.parametrize("script", list(SCRIPTS))
def test_many_short_intervals(script, fixed, monkeypatch):
    rng = np.random.default_rng(fixed)
    dims = [(32, 32), (8, 8), (200, 33), (31, 33)]
    with pcr_synth.scan_script(SCRIPTS[script]):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), d, t) for (w, h), d, t in zip(dims, (0.15, 1.0, 0.3, 0.02), (60, 1023, 100, 500))]
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=fixed == 0, restart_fixed=fixed)
    monkeypatch.setenv("PCR_PACK_WARPS", str(1 << 20))
    monkeypatch.setenv("PCR_SHORT_WARPS", "0")
    _compare(rec, (1, 5) if script == "ten" else range(1, len(SCRIPTS[script]) + 1))

"""The restart-interval index with a warp per scan and with a CTA per scan (PCR_INDEX_CTAS, read when a record is opened, chooses):
scans of a few bytes to many tiles of 512, so that runs of tiles begin and end at every remainder of a word, with stuffed zeros
and markers anywhere."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from test_gpu_kernel_edges import _compare, _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [0, 1 << 20])
@pytest.mark.parametrize("fixed", [None, 0, 1, 9])
@pytest.mark.parametrize("script", ["ten", "baseline"])
def test_runs_of_tiles(script, fixed, ctas, monkeypatch):
    """fixed: MCUs an interval (None: no markers, 0: a row)."""
    rng = np.random.default_rng(17 + (fixed or 0))
    dims = [(8, 8), (40, 24), (72, 40), (136, 56), (104, 104), (200, 72), (264, 200), (24, 400)]
    with pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE if script == "baseline" else None):
        coeffs = [_field(rng, pcr_synth.num_blocks(w, h), float(rng.uniform(0.05, 0.9)), 1023) for w, h in dims]
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=fixed == 0, restart_fixed=fixed or 0)
    monkeypatch.setenv("PCR_INDEX_CTAS", str(ctas))
    _compare(rec, (1,) if script == "baseline" else (1, 10))

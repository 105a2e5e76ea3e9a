"""The places where the kernels' decompositions change: numbers of restart intervals around a warp's halves, the order in
which fidelities are decoded, coefficients at the corner the short transform is made for, scans around the size that is
staged in shared memory, and the table of images.  Everything against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import pcr_synth
from oracle import pcr_oracle as O

pytestmark = pytest.mark.gpu


def _compare(rec, ks):
    import torch
    from paper_1911_00472_b200 import Decoder, pcr_image_blocks
    dec = Decoder(rec.bytes)
    try:
        for k in ks:
            out = dec.decode(k)
            torch.cuda.synchronize()
            assert dec.status() == (-1, 0), k
            pixels, coeffs = out.cpu().numpy(), dec.coeffs().cpu().numpy()
            for i in range(rec.n_images):
                want_c, want = O.decode_image(rec.bytes, i, k)
                inf = dec.info[i]
                a, b = pcr_image_blocks(dec.handle, i)
                assert np.array_equal(coeffs[a:a + b], want_c), (k, i)
                assert np.array_equal(pixels[inf.out_offset:inf.out_offset + inf.out_bytes].reshape(want.shape), want), (k, i)
    finally:
        dec.close()


def _field(rng, n_blocks, density, top):
    c = np.where(rng.random((n_blocks, 64)) < density, rng.integers(-top, top + 1, (n_blocks, 64)), 0)
    c[:, 0] = rng.integers(-500, 501, n_blocks)
    return c.astype(np.int16)


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 32, 33])
def test_intervals_around_a_warp(rows):
    """Luminance scans of 1..33 restart intervals per image (pairs of refinements take sixteen of them, other items 32),
    three images behind one another so that items run on from one to the next; wide enough for several top-ups."""
    rng = np.random.default_rng(rows)
    dims = [(72, 8 * rows), (9, 8 * rows), (136, 8 * max(1, rows - 1))]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), d, 40) for (w, h), d in zip(dims, (0.3, 0.05, 0.6))]
    _compare(pcr_synth.record_from_coeffs(dims, coeffs), (1, 2, 5, 6, 9, 10))


@pytest.mark.parametrize("restart_rows", [True, False])
def test_fidelity_lowered_on_one_handle(restart_rows):
    """What a decode at high fidelity leaves behind (refined DC bits, values of later scans) does not show in a
    later one at lower fidelity; DC scans of single components, so that a component may have none yet."""
    script = [((0,), 0, 0, 0, 1), ((1,), 0, 0, 0, 0), ((0,), 1, 63, 0, 1), ((2,), 0, 0, 0, 1), ((0,), 0, 0, 1, 0),
              ((2,), 0, 0, 1, 0), ((1,), 1, 63, 0, 0), ((2,), 1, 5, 0, 0), ((0,), 1, 63, 1, 0)]
    rng = np.random.default_rng(3)
    dims = [(50, 41), (17, 96)]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), 0.2, 9) for w, h in dims]
    with pcr_synth.scan_script(script):
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=restart_rows)
    _compare(rec, range(len(script), 0, -1))


@pytest.mark.parametrize("largest", [(192, 128), (400, 390)])
@pytest.mark.parametrize("single", [True, False])
def test_dc_refinement_beside_ac_refinement(largest, single):
    """DC refinements in the blocks behind a wave's restart intervals: images of 1, 95, 96, 97 and 625 MCUs (a block takes 96
    at a time, one or two blocks an image), one interleaved scan or one for each component, and the last one alone in its
    wave."""
    dc = [((c,), 0, 0, 2, 1) for c in range(3)] if single else [((0, 1, 2), 0, 0, 2, 1)]
    script = [((0, 1, 2), 0, 0, 0, 2), ((0,), 1, 63, 0, 1), ((1,), 1, 63, 0, 0), ((2,), 1, 63, 0, 0)] + dc + [
        ((0,), 1, 63, 1, 0), ((0, 1, 2), 0, 0, 1, 0)]
    rng = np.random.default_rng(5)
    dims = [largest, (16, 16), (19 * 16, 75), (97 * 16, 9)]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), 0.1, 9) for w, h in dims]
    with pcr_synth.scan_script(script):
        rec = pcr_synth.record_from_coeffs(dims, coeffs)
    _compare(rec, range(len(script) - len(dc) - 1, len(script) + 1))


@pytest.mark.parametrize("outside", [None, (4, 0), (0, 4), (7, 7)])
@pytest.mark.parametrize("samp", [(2, 2, 3), (1, 1, 3), (1, 1, 1)])
def test_corner_transform(outside, samp):
    """Coarse scans whose coefficients fill the low 4x4 corner of every block, to the corner's own limit (3, 3), and
    the same with one coefficient outside it in one block: the warp that holds the block takes the full transform."""
    nat = {int(n): z for z, n in enumerate(pcr_synth.zigzag())}
    rng = np.random.default_rng(11)
    with pcr_synth.sampling(*samp):
        dims = [(130, 70), (33, 31)]
        coeffs = []
        for w, h in dims:
            c = np.zeros((pcr_synth.num_blocks(w, h), 64), dtype=np.int16)
            for r in range(4):
                for q in range(4):
                    c[:, nat[8 * r + q]] = rng.integers(-60, 61, c.shape[0])
            if outside is not None:
                c[len(c) // 3, nat[8 * outside[0] + outside[1]]] = 44
            coeffs.append(c)
        rec = pcr_synth.record_from_coeffs(dims, coeffs)
    groups = 3 if samp[2] == 1 else 5            # the coarse scans of the script
    _compare(rec, (groups - 1, groups))


@pytest.mark.parametrize("script", ["ten", "baseline"])
@pytest.mark.parametrize("density", [0.02, 0.12, 0.5])
def test_long_scans_around_the_staged_size(script, density):
    """Scans without restart markers from a few hundred bytes to several times the words that are staged."""
    rng = np.random.default_rng(int(100 * density))
    dims = [(264, 200), (40, 24), (8, 8)]
    coeffs = [_field(rng, pcr_synth.num_blocks(w, h), density, 60) for w, h in dims]
    with pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE if script == "baseline" else None):
        rec = pcr_synth.record_from_coeffs(dims, coeffs, restart_rows=False)
    _compare(rec, (1,) if script == "baseline" else (1, 5, 10))


def test_image_table(rec1_small):
    from paper_1911_00472_b200 import Decoder, binding
    dec = Decoder(rec1_small.bytes)
    try:
        some = binding.pcr_get_images(dec.handle, 2, 3)
        for j, inf in enumerate(some):
            one = binding.pcr_get_image(dec.handle, 2 + j)
            assert (inf.width, inf.height, inf.label, inf.out_offset, inf.out_bytes) == (one.width, one.height, one.label, one.out_offset, one.out_bytes)
        assert len(dec.info) == dec.n_images
        for first, count in ((-1, 1), (0, dec.n_images + 1), (dec.n_images, 1)):
            with pytest.raises(binding.PcrError):
                binding.pcr_get_images(dec.handle, first, count)
    finally:
        dec.close()

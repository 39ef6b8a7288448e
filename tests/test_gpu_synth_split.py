"""Small synthesis launches (a probe's rows over a cluster of 4 or 2 CTAs) against large ones (one
CTA per probe): the same sums in the same order, so every readout of a sub-region equals, bit for
bit, that part of the readout of the whole region. 36 and 37 probes lie at the line between
clusters of four and of two, 76 and 77 at the one to the large form (on 152 SMs); the spacings give
even and odd placements, and L leaves a rest in the batches of 2 and 5 waves.
"""
import dataclasses

import numpy as np
import pytest

from paper_2310_16829_gb300 import lma, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,precision,L", [(128, WL.PREC_C64, 32), (128, WL.PREC_FP16_STORE, 13), (64, WL.PREC_C64, 12),
                                                (256, WL.PREC_C64, 1)])
@pytest.mark.parametrize("spacing", [4, 5])
def test_small_launches_read_the_same_as_large_ones(window, precision, L, spacing):
    w = WL.perovskite_workload(cells=5, nx=256, n_slices=2, n_phonons=1, seed_base=720)
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    basis = lma.Basis(ctx, spec, w.probe, dataclasses.replace(w.basis, window=window, precision=precision, L=L))
    nx, ny = 22, 9
    det = [WL.Detector(0.0, 0.02), WL.Detector(0.03, 0.06)]
    region = lambda x, y, w_, h: WL.Region(7 + spacing * x, 250 + spacing * y, w_, h, (spacing, spacing))  # noqa: E731
    whole = region(0, 0, nx, ny)
    image, rings = basis.image(det, whole), basis.image_rings(0.01, 5, whole)
    pattern = basis.image_4d(7, 5, whole)
    assert np.all(np.isfinite(image)) and image.max() > 0
    for x, y, pw, ph in ((0, 0, 1, 1), (3, 2, 6, 6), (2, 1, 18, 2), (0, 3, 19, 2), (3, 0, 19, 4), (0, 0, 11, 7)):
        part = region(x, y, pw, ph)
        assert np.array_equal(basis.image(det, part), image[:, y:y + ph, x:x + pw]), (pw, ph)
    part = region(3, 2, 6, 6)
    assert np.array_equal(basis.image_rings(0.01, 5, part), rings[:, 2:8, 3:9])
    assert np.array_equal(basis.image_4d(7, 5, part), pattern[2:8, 3:9])
    part = region(1, 1, 19, 2)
    assert np.array_equal(basis.image_rings(0.01, 5, part), rings[:, 1:3, 1:20])
    assert np.array_equal(basis.image_4d(7, 5, part), pattern[1:3, 1:20])

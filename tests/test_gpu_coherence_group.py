"""Four probe variants in one synthesis launch against one launch per variant: with all weight on one
variant the average is that variant's image, so both calls give the same bits. Five variants leave
one for the per-variant launch; L = 13 and 1 leave a rest in the batches of two waves; the
spacings give even and odd placements.
"""
import dataclasses

import numpy as np
import pytest

from paper_2310_16829_gb300 import lma, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,precision,L", [(128, WL.PREC_C64, 32), (128, WL.PREC_FP16_STORE, 13), (64, WL.PREC_C64, 12),
                                                (256, WL.PREC_C64, 1)])
@pytest.mark.parametrize("spacing", [4, 5])
def test_four_variants_at_once_equal_one_by_one(window, precision, L, spacing):
    w = WL.perovskite_workload(cells=5, nx=256, n_slices=2, n_phonons=2, seed_base=740)
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    basis = lma.Basis(ctx, spec, w.probe, dataclasses.replace(w.basis, window=window, precision=precision, L=L))
    det = [WL.Detector(0.0, 0.02), WL.Detector(0.03, 0.06)]
    region = WL.Region(7, 250, 13, 7, (spacing, spacing))
    foci = (-40.0, -15.0, 0.0, 25.0, 60.0)
    seen = []
    for k, dz in enumerate(foci):
        series = [(f, 0.0, 1.0 if i == k else 0.0) for i, f in enumerate(foci)]
        one = basis.image_coherent([(dz, 0.0, 1.0)], det, region)
        assert np.array_equal(basis.image_coherent(series, det, region), one), (k, dz)
        assert np.all(np.isfinite(one)) and one.max() > 0
        seen.append(one)
    assert any(not np.array_equal(seen[0], s) for s in seen[1:])

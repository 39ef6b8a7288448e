"""Column edits where the propagation window is not 128 pixels: an edit marks those exit waves stale
whose own window meets the touched pixels, on both axes. The number marked is counted here pixel by
pixel; waves 105 to 148 pixels from the column (which only windows of 256 pixels reach, along x or
along y) are, after the next image, those of a specimen built with the edited atoms, bit for bit.
"""
import dataclasses

import numpy as np
import pytest

from oracle import lma_oracle as O
from paper_2310_16829_gb300 import lma, workloads as WL

pytestmark = pytest.mark.gpu


def _touched(w, cx, cy, r_site):
    """Per axis, the grid pixels within r_cut of a touched atom, with one pixel of margin."""
    g, r_cut = w.grid, w.potential.r_cut
    ddx = np.concatenate([at.x - cx for at in w.phonons])
    ddy = np.concatenate([at.y - cy for at in w.phonons])
    ddx -= g.lx * np.rint(ddx / g.lx)
    ddy -= g.ly * np.rint(ddy / g.ly)
    hit = ddx ** 2 + ddy ** 2 < r_site ** 2
    out = []
    for c, dd, step, n in ((cx, ddx[hit], g.dx, g.nx), (cy, ddy[hit], g.dy, g.ny)):
        lo = int(np.floor((c + dd.min() - r_cut) / step)) - 1
        hi = int(np.ceil((c + dd.max() + r_cut) / step)) + 1
        out.append(set(np.arange(lo, hi + 1) % n))
    return out


@pytest.mark.parametrize("window", [64, 128, 256])
@pytest.mark.parametrize("px,py", [(140, 276), (276, 140), (412, 276)])
def test_edit_renews_the_waves_whose_window_meets_it(window, px, py):
    w = WL.perovskite_workload(cells=10, nx=512, n_slices=2, n_phonons=1, seed_base=3110)
    w = dataclasses.replace(w, basis=dataclasses.replace(w.basis, window=window, L=4))
    region = WL.Region(px, py, 3, 3, (4, 4))
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    basis = lma.Basis(ctx, spec, w.probe, w.basis)
    basis.propagate(0)
    translates = sorted({int(i) for a in range(3) for b in range(3)
                         for i in basis.coefficients(px + 4 * a, py + 4 * b)[2]})
    before = {i: basis.exit_wave(i) for i in translates}
    cx, cy = 5.5 * WL.ABO3_A, 5.5 * WL.ABO3_A           # pixel 281.6 on both axes
    changed, stale = spec.edit_column(basis, cx, cy, 0.5, lma.LMA_EDIT_SET_SPECIES, 2)
    assert changed > 0
    counts = []
    for n, pixels in zip((512, 512), _touched(w, cx, cy, 0.5)):
        counts.append(sum(1 for p in range(2, n, 4)
                          if any((p - window // 2 + k) % n in pixels for k in range(window))))
    assert stale == counts[0] * counts[1], (window, stale, counts)
    basis.image(w.detectors, region)
    ph = []
    for at in w.phonons:
        x, y, s, sp, _ = O.edit_column(at.x, at.y, at.slice, at.species, w.grid.lx, w.grid.ly, cx, cy, 0.5, 1, 2)
        ph.append(WL.Atoms(x, y, s, sp))
    spec2 = lma.Specimen(ctx, w.grid, w.potential, ph)
    full = lma.Basis(ctx, spec2, w.probe, w.basis)
    full.propagate(0)
    for i in translates:
        got = basis.exit_wave(i)
        assert np.array_equal(got, full.exit_wave(i)), (window, px, py, i)
        assert np.array_equal(got, before[i]) == (window != 256), (window, px, py, i)

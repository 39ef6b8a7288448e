"""3D and 4D readouts where the propagation window W is not the detection window D = 128: rings and
patterns are taken on the D x D spectrum inside the bandlimit of that grid (radius 42 pixels at 2/3,
where W = 64 has 21 and W = 256 has 85). Against the FP64 oracle with the bounds of
``parity_floor``, for few probes and for more than a cluster launch takes.
"""
import dataclasses

import numpy as np
import pytest

from oracle import lma_oracle as O
from paper_2310_16829_gb300 import lma, workloads as WL
from parity_floor import assert_floor, oracles

pytestmark = pytest.mark.gpu


def _objects(window):
    w = WL.perovskite_workload(cells=5, nx=256, n_slices=4, n_phonons=1, seed_base=2310)
    w = dataclasses.replace(w, basis=dataclasses.replace(w.basis, window=window, L=12))
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    return w, lma.Basis(ctx, spec, w.probe, w.basis)


def _probes(region, w):
    return O.region_probes(region.px0, region.py0, region.npx, region.npy, region.spacing_px, w.grid.nx, w.grid.ny)


@pytest.mark.parametrize("window", [64, 256])
def test_rings_of_other_windows_match_oracle(window):
    w, basis = _objects(window)
    few, many = WL.Region(250, 12, 2, 2, (4, 4)), WL.Region(250, 12, 13, 6, (4, 4))
    got = basis.image_rings(0.01, 9, few)                # up to 90 mrad, 44 pixels
    orc, emu = oracles(w)
    ref, e = orc.image_rings(0.01, 9, _probes(few, w)), emu.image_rings(0.01, 9, _probes(few, w))
    assert np.all(ref[:8] > 0)
    assert_floor(got.reshape(9, -1), ref, e, label=f"rings W={window}")
    assert np.array_equal(basis.image_rings(0.01, 9, many)[:, :2, :2], got)


@pytest.mark.parametrize("window", [64, 256])
def test_patterns_of_other_windows_match_oracle(window):
    w, basis = _objects(window)
    few, many = WL.Region(250, 12, 2, 1, (4, 4)), WL.Region(250, 12, 13, 6, (4, 4))
    A, B = 50, 45
    got = basis.image_4d(A, B, few)
    orc, emu = oracles(w)
    ref, e = orc.image_4d(A, B, _probes(few, w)), emu.image_4d(A, B, _probes(few, w))
    ia, ib = np.arange(-A, A + 1), np.arange(-B, B + 1)
    band = 9 * (ia[None, :] ** 2 + ib[:, None] ** 2) <= w.basis.det_window ** 2
    assert np.all(ref[:, ~band] == 0.0)
    for g, r, ee in zip(got.reshape(2, 2 * B + 1, 2 * A + 1).astype(np.float64), ref, e):
        assert_floor(g.reshape(1, -1), r.reshape(1, -1), ee.reshape(1, -1), label=f"pattern W={window}")
    assert np.array_equal(basis.image_4d(A, B, many)[:1, :2], got)

"""The W = 256 slice kernel for bandlimit radii up to 85 pixels, at the edges of its rule and of its
window placement, against the FP64 oracle: radius 85 (2/3 of Nyquist) and 86 (the general kernel),
odd window origins (8-byte staging), windows whose halves wrap around the cell on both axes, and a
translate count that leaves SMs without work. Exit waves to 5e-5 of their peak, as in
``test_gpu_windows``.
"""
import dataclasses

import numpy as np
import pytest

from paper_2310_16829_gb300 import lma, workloads as WL
from parity_floor import oracles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frac", [2.0 / 3.0, 0.675])
@pytest.mark.parametrize("offset,nx", [(2, 256), (1, 256), (3, 512)])
def test_exit_waves_match_oracle(frac, offset, nx):
    w = WL.perovskite_workload(cells=nx // 50, nx=nx, n_slices=3, n_phonons=1, seed_base=2950)
    w = dataclasses.replace(w, grid=dataclasses.replace(w.grid, bandlimit_frac=frac),
                            basis=dataclasses.replace(w.basis, window=256, f=8, L=4, in_offset_px=(offset, offset)))
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    basis = lma.Basis(ctx, spec, w.probe, w.basis)
    basis.propagate(0)
    orc, _ = oracles(w)
    n = basis.info().n_translates
    for i in (0, n // 2 + 3, n - 1):
        got, ref = basis.exit_wave(i), orc.exit_wave(0, i)
        assert np.max(np.abs(got - ref)) < 5e-5 * np.max(np.abs(ref)), (frac, offset, nx, i)

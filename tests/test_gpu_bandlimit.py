"""Narrow bandlimits: every slice kernel at radii far below the 2/3 that the default grid has, against
the FP64 oracle. In the 128-pixel kernels a warp whose columns all lie outside the band skips the
propagation of them; below radius 32 (fraction 0.5) more than one warp of a group does, and at
fraction 0.02 (radius 1) all but those of the central columns. Exit waves to 5e-5 of their peak
as in ``test_gpu_parity`` (the FP16 store: plus its rounding, 2^-11 of a component and 2^-23 of
the largest); readings of complex64 waves to the bounds of ``parity_floor``.
"""
import dataclasses

import numpy as np
import pytest

from oracle import lma_oracle as O
from paper_2310_16829_gb300 import lma, workloads as WL
from parity_floor import assert_floor, oracles

pytestmark = pytest.mark.gpu

FRACS = [0.02, 0.1, 0.3, 0.49, 0.5, 2.0 / 3.0]


def _workload(frac, window, precision, offset):
    w = WL.perovskite_workload(cells=5, nx=256, n_slices=4, n_phonons=1, seed_base=2960)
    return dataclasses.replace(w, grid=dataclasses.replace(w.grid, bandlimit_frac=frac),
                               basis=dataclasses.replace(w.basis, window=window, precision=precision,
                                                         in_offset_px=(offset, offset)))


def _assert_wave(got, ref, half, label):
    peak = np.max(np.abs(ref))
    if not half:
        assert np.max(np.abs(got - ref)) < 5e-5 * peak, (label, np.max(np.abs(got - ref)) / peak)
        return
    m = np.max(np.abs(np.stack([ref.real, ref.imag])))
    for a, b in ((got.real, ref.real), (got.imag, ref.imag)):
        assert np.all(np.abs(a - b) <= 2.0 ** -11 * np.abs(b) + 2.0 ** -23 * m + 5e-5 * peak), label


def _check(frac, window, precision, offset):
    w = _workload(frac, window, precision, offset)
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    orc, emu = oracles(w)
    half = precision == WL.PREC_FP16_STORE
    whole = lma.Basis(ctx, spec, w.probe, w.basis)     # every translate in one launch
    whole.propagate(0)
    n = whole.info().n_translates
    for i in (0, 64 * 32 + 17, n - 1):
        _assert_wave(whole.exit_wave(i), orc.exit_wave(0, i), half, (frac, window, precision, offset, i))
    few = lma.Basis(ctx, spec, w.probe, w.basis)       # the translates of six probes only
    region = WL.Region(250, 60, 3, 2, (4, 4))
    dets = [WL.Detector(0.0, 0.01), WL.Detector(0.0, 0.2)]
    img = few.image(dets, region).reshape(2, -1)
    assert np.all(np.isfinite(img))
    i = int(few.coefficients(region.px0, region.py0)[2][0])
    _assert_wave(few.exit_wave(i), orc.exit_wave(0, i), half, (frac, window, precision, offset, "few", i))
    if half:
        return
    probes = O.region_probes(region.px0, region.py0, 3, 2, region.spacing_px, w.grid.nx, w.grid.ny)
    tol = 1e-4 if precision == WL.PREC_C64 else 1e-3   # the contracts of the precision forms
    assert_floor(img, orc.image(dets, probes), emu.image(dets, probes), tol=tol, label=f"{frac} {window} {precision}")


@pytest.mark.parametrize("frac", FRACS)
@pytest.mark.parametrize("offset", [1, 2])
@pytest.mark.parametrize("precision", [WL.PREC_C64, WL.PREC_FP16_STORE])
def test_narrow_bandlimits_match_oracle(frac, offset, precision):
    _check(frac, 128, precision, offset)


@pytest.mark.parametrize("frac", [0.1, 0.3, 0.49])
@pytest.mark.parametrize("window", [64, 256])
def test_narrow_bandlimits_of_other_windows_match_oracle(window, frac):
    _check(frac, window, WL.PREC_C64, 1 if frac == 0.3 else 2)


@pytest.mark.parametrize("frac", FRACS)
@pytest.mark.parametrize("offset", [1, 2])
def test_narrow_bandlimits_on_tensor_cores_match_oracle(frac, offset):
    _check(frac, 128, WL.PREC_MIXED, offset)

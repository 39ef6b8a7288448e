"""The W = 64 slice kernels against each other: a list of at most one translate per SM takes the
512-thread kernel, longer ones two translates per 128-thread CTA. Both run the same transforms in
the same order, so the exit waves are equal bit for bit; the 512-thread kernel is held to the
oracle by ``test_gpu_windows``.
"""
import dataclasses

import numpy as np
import pytest

from paper_2310_16829_gb300 import lma, workloads as WL

pytestmark = pytest.mark.gpu


# 2/3 and 0.685: the pruned kernel (radius below 22 pixels); 0.69 and 1.0: above it. Offset 1 gives
# odd window origins (8-byte staging). nax x nay = 64 x 32 translates, or 13 x 32 / 16 with spacing
# 20 and 16 (an odd count: the last translate of the list is alone in its CTA).
@pytest.mark.parametrize("frac", [2.0 / 3.0, 0.685, 0.69, 1.0])
@pytest.mark.parametrize("offset", [1, 2])
def test_long_and_short_lists_give_the_same_exit_waves(frac, offset):
    w = WL.perovskite_workload(cells=5, nx=256, n_slices=3, n_phonons=1, seed_base=700)
    w = dataclasses.replace(w, grid=dataclasses.replace(w.grid, bandlimit_frac=frac),
                            basis=dataclasses.replace(w.basis, window=64, L=12, in_offset_px=(offset, offset)))
    ctx = lma.Context(0)
    spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
    long = lma.Basis(ctx, spec, w.probe, w.basis)
    long.propagate(0)
    short = lma.Basis(ctx, spec, w.probe, w.basis)
    region = WL.Region(120, 40, 3, 3, (8, 8))          # under 100 translates
    short.image(w.detectors, region)
    seen = 0
    for b in range(region.npy):
        for a in range(region.npx):
            _, _, translates, _ = short.coefficients(region.px0 + 8 * a, region.py0 + 8 * b)
            for i in translates:
                x, y = short.exit_wave(int(i)), long.exit_wave(int(i))
                assert np.array_equal(x, y), (frac, offset, int(i))
                assert np.all(np.isfinite(x)) and np.max(np.abs(x)) > 0
                seen += 1
    assert seen == 9 * 12


def test_an_odd_list_stores_every_wave_once():
    """153 to 255 translates of two specimens in one launch, both counts odd."""
    ws = [WL.perovskite_workload(cells=5, nx=256, n_slices=ns, n_phonons=1, seed_base=710 + ns) for ns in (2, 4)]
    ctx = lma.Context(0)
    bases, regions, outs = [], [], []
    for k, w in enumerate(ws):
        spec = lma.Specimen(ctx, w.grid, w.potential, w.phonons)
        bases.append(lma.Basis(ctx, spec, w.probe, dataclasses.replace(w.basis, window=64, L=9)))
        regions.append(WL.Region(16, 20, 9, 7 + 2 * k, (4, 4)))
        outs.append(np.empty((1, 7 + 2 * k, 9)))
    lma.image_many(ctx, bases, ws[0].detectors, regions, outs)
    for w, region, out in zip(ws, regions, outs):
        one = np.empty_like(out)
        alone = lma.Context(0)
        spec = lma.Specimen(alone, w.grid, w.potential, w.phonons)
        basis = lma.Basis(alone, spec, w.probe, dataclasses.replace(w.basis, window=64, L=9))
        for b in range(region.npy):                       # one row of probes at a time: short lists
            row = WL.Region(region.px0, region.py0 + 4 * b, region.npx, 1, (4, 4))
            one[:, b:b + 1] = basis.image(w.detectors, row)
        assert np.array_equal(out, one)

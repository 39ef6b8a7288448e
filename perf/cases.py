"""The imaging calls whose speed this library is measured by, with their inputs and exact results.

Each case is one call (or one short request) that a program makes through the public binding
``paper_2310_16829_gb300.lma``: full images, reading probes out of resident exit waves, column
edits, focal series, 4D patterns, batches of small specimens, and images of atoms that have just
changed on the host. Specimens are layered crystals with seeded frozen-phonon displacements.

``exact`` restates the method (potential, multislice of the lattice translates, least-squares
coefficients, synthesis, detectors) in 64 bits with torch and numpy alone.
"""
from __future__ import annotations

import math
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2310_16829_gb300 import lma, workloads as WL  # noqa: E402

D = 128                       # detection window of the library
GAUSS_ALPHA = 0.025           # probe aperture (rad) of the layered crystals
PEAKS = WL.ABO3_PEAKS
TERM_FRAC, TERM_WIDTH, R_CUT = (0.7, 0.3), (0.15, 0.5), 3.0
RMS = 0.08                    # phonon displacement (Angstrom)
HAADF = (0.070, 0.200)
BRIGHT = (0.0, 0.020)
ANNULI = (BRIGHT, (0.012, 0.025), (0.025, 0.070), HAADF)   # bright field, annular bright and dark field, HAADF
# (fractional x, fractional y, species) of the two alternating layers of ABO3 along [001]
LAYERS = (((0.0, 0.0, 0), (0.5, 0.5, 2)), ((0.5, 0.5, 1), (0.5, 0.0, 2), (0.0, 0.5, 2)))


def _case(name=None, **kw):
    c = dict(kind="image", nx=512, ny=512, cells_x=10, cells_y=10, slices=50, configs=1, window=128,
             precision="c64", L=32, f=1, in_spacing=4, in_offset=2, npx=128, npy=128, spacing_x=4, spacing_y=4,
             px0=0, py0=0, detector="haadf", defocus=0.0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # Live view: a few probes read out of exit waves that are already resident. The smallest
        # call: launches and host work.
        _case("live_view_8x8", kind="readout", nx=256, ny=256, cells_x=5, cells_y=5, slices=20, npx=8, npy=8,
              spacing_x=16, spacing_y=16, px0=60, py0=60, detector="all"),
        # A small periodic cell, W equal to the grid: the whole image of a unit cell study.
        _case("unit_cell_128", nx=128, ny=128, cells_x=2, cells_y=2, slices=10, npx=32, npy=32),
        # The benchmark: 100 A of ABO3, 8 frozen phonons, 128 x 128 HAADF pixels.
        _case("benchmark_512_8ph", configs=8),
        # An odd scan: probe steps that do not divide the grid (many coefficient classes), an odd
        # corner and an odd lattice offset, a rectangular specimen, two phonons.
        _case("odd_scan_256x512", nx=256, ny=512, cells_x=5, cells_y=10, slices=30, configs=2, npx=37, npy=83,
              spacing_x=5, spacing_y=6, px0=3, py0=7, in_offset=1, L=37),
        # A column changed in a resident 200 A specimen and its surroundings imaged again, for two
        # columns: an editing session. Results go to the host.
        _case("column_edit_1024", kind="edit", nx=1024, ny=1024, cells_x=20, cells_y=20, slices=100, npx=64, npy=64),
        # Focal series (partial coherence): five probes read out from one set of resident waves.
        _case("focal_series_512", kind="focal", slices=25, npx=128, npy=128),
        # 4D STEM: the diffraction patterns inside the bandlimit, for a denoiser or ptychography.
        _case("patterns_4d_256", kind="pattern", nx=256, ny=256, cells_x=5, cells_y=5, slices=20, configs=2, npx=48,
              npy=48, half=42),
        # Narrow propagation windows: fast surveys of thin specimens.
        _case("window_64_512", window=64),
        # Wide propagation windows: thick specimens whose high-angle scattering leaves 128 pixels.
        _case("window_256_512", window=256, slices=20),
        # Tensor-core transforms.
        _case("mixed_256", nx=256, ny=256, cells_x=5, cells_y=5, slices=20, configs=2, npx=64, npy=64, precision="mixed"),
        # Half-size store of the exit waves with a bright-field readout: large scans in less memory.
        _case("fp16_store_bright_512", slices=20, npx=101, npy=77, spacing_x=5, spacing_y=6, precision="fp16",
              detector="bright"),
        # New atom positions from the host (a relaxation or fitting loop), image back on the host.
        _case("fresh_atoms_256", kind="fresh", nx=256, ny=256, cells_x=5, cells_y=5, slices=40, configs=2, npx=64, npy=64),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["image", "image", "image", "readout", "focal", "pattern", "fresh", "edit"])
        nx, ny = rng.choice([128, 256, 256, 512]), rng.choice([128, 256, 256, 512])
        window, precision = 128, "c64"
        if kind == "image":
            window = rng.choice([64, 128, 128, 128, 256])
            if window == 128:
                precision = rng.choice(["c64", "c64", "fp16", "mixed"])
        nx, ny = max(nx, window), max(ny, window)
        c = _case(kind=kind, nx=nx, ny=ny, cells_x=max(2, nx * 10 // 512), cells_y=max(2, ny * 10 // 512),
                  slices=log(4, 100), configs=rng.choice([1, 1, 2, 3]) if kind != "edit" else 1, window=window,
                  precision=precision, L=rng.randint(12, 60), f=rng.choice([1, 1, 2]), in_offset=rng.randint(0, 3),
                  npx=log(5, 128), npy=log(5, 128), spacing_x=rng.randint(2, 9), spacing_y=rng.randint(2, 9),
                  px0=rng.randrange(nx), py0=rng.randrange(ny), defocus=round(rng.uniform(-60.0, 60.0), 1))
        if kind in ("readout", "focal"):
            c["detector"] = rng.choice(["haadf", "all"])
        if kind == "readout":
            c["npx"], c["npy"] = rng.randint(3, 24), rng.randint(3, 24)
        if kind == "edit":
            c["npx"] = c["npy"] = rng.randint(24, 64)
            c["spacing_x"] = c["spacing_y"] = 4
            if min(nx, ny) < 256:
                continue
        if kind == "pattern":
            c["half"] = rng.randint(8, 63)
            c["npx"], c["npy"] = min(c["npx"], 40), min(c["npy"], 40)
        if precision == "fp16":
            c["detector"] = "bright"
        if _translates(c) * c["slices"] * c["configs"] * (window / 128) ** 2 <= 1.0e6:
            return c


def _translates(c):
    s = c["in_spacing"] * c["f"]
    return (c["nx"] // s) * (c["ny"] // s)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _grid(c):
    return WL.Grid(nx=c["nx"], ny=c["ny"], lx=c["cells_x"] * WL.ABO3_A, ly=c["cells_y"] * WL.ABO3_A, slice_dz=2.0,
                   n_slices=c["slices"], lam=WL.LAMBDA_300KV, sigma=WL.SIGMA_300KV)


def _crystals(c, seed):
    """One atom list per frozen-phonon configuration, displaced by the seed."""
    rng = np.random.default_rng(seed)
    ii = np.tile(np.arange(c["cells_x"], dtype=np.float64), c["cells_y"])
    jj = np.repeat(np.arange(c["cells_y"], dtype=np.float64), c["cells_x"])
    xs, ys, ss, sp = [], [], [], []
    for s in range(c["slices"]):
        for fx, fy, kind in LAYERS[s % 2]:
            xs.append((ii + fx) * WL.ABO3_A)
            ys.append((jj + fy) * WL.ABO3_A)
            ss.append(np.full(ii.shape, s, np.int32))
            sp.append(np.full(ii.shape, kind, np.int16))
    x, y, s, sp = (np.concatenate(v) for v in (xs, ys, ss, sp))
    out = []
    for _ in range(c["configs"]):
        d = rng.normal(0.0, RMS, size=(2, x.shape[0]))
        out.append(WL.Atoms(x + d[0], y + d[1], s, sp))
    return out


def _edit_columns(c, seed):
    """Two A-site columns (one species through the whole thickness), well apart."""
    rng = np.random.default_rng(seed + 1)
    i, j = int(rng.integers(0, c["cells_x"])), int(rng.integers(0, c["cells_y"]))
    k, m = (i + c["cells_x"] // 2) % c["cells_x"], (j + c["cells_y"] // 2) % c["cells_y"]
    return [(i * WL.ABO3_A, j * WL.ABO3_A), (k * WL.ABO3_A, m * WL.ABO3_A)]


def _regions(c, seed):
    if c["kind"] != "edit":
        return [WL.Region(c["px0"], c["py0"], c["npx"], c["npy"], (c["spacing_x"], c["spacing_y"]))]
    g, out = _grid(c), []
    for cx, cy in _edit_columns(c, seed):
        px, py = int(round(cx / g.dx)) // 4 * 4, int(round(cy / g.dy)) // 4 * 4
        out.append(WL.Region(px - c["npx"] // 2 * 4, py - c["npy"] // 2 * 4, c["npx"], c["npy"], (4, 4)))
    return out


def _annuli(c):
    return {"haadf": (HAADF,), "bright": (BRIGHT,), "all": ANNULI}[c["detector"]]


def _focal(c):
    """(defocus, C_s, weight) of a five-step focal series around the case's focus."""
    return [(c["defocus"] + d, 0.0, w) for d, w in ((-40.0, 0.1), (-20.0, 0.25), (0.0, 0.3), (20.0, 0.25), (40.0, 0.1))]


def prepare(case, seed):
    c = case
    precision = {"c64": lma.LMA_PREC_C64, "fp16": lma.LMA_PREC_FP16_STORE, "mixed": lma.LMA_PREC_MIXED}[c["precision"]]
    ctx = lma.Context(0)
    atoms = _crystals(c, seed)
    pot = WL.Potential(peak=PEAKS, term_frac=TERM_FRAC, term_width=TERM_WIDTH, r_cut=R_CUT)
    spec = lma.Specimen(ctx, _grid(c), pot, atoms)
    desc = WL.BasisDesc(in_spacing_px=(c["in_spacing"],) * 2, in_offset_px=(c["in_offset"],) * 2, f=c["f"], L=c["L"],
                        window=c["window"], precision=precision)
    basis = lma.Basis(ctx, spec, WL.Probe(alpha_max=GAUSS_ALPHA, defocus=c["defocus"]), desc)
    regions, det = _regions(c, seed), [WL.Detector(*a) for a in _annuli(c)]
    st = {"case": c, "basis": basis, "spec": spec, "regions": regions, "det": det, "atoms": atoms}
    n = (c["npy"], c["npx"])
    if c["kind"] == "pattern":
        p = 2 * c["half"] + 1
        st["out"] = torch.empty(n + (p, p), dtype=torch.float32, device="cuda:0")
    elif c["kind"] not in ("edit", "fresh"):
        st["out"] = torch.empty((len(det),) + n, dtype=torch.float64, device="cuda:0")
    if c["kind"] in ("readout", "focal"):
        basis.image(det, regions[0], out=st["out"])            # the waves that the readout finds resident
    elif c["kind"] == "edit":
        st["columns"] = _edit_columns(c, seed)
        basis.propagate(0)
    return st


def run(state):
    c, basis, det = state["case"], state["basis"], state["det"]
    if c["kind"] == "readout":
        return basis.image(det, state["regions"][0], out=state["out"])
    if c["kind"] == "focal":
        return basis.image_coherent(_focal(c), det, state["regions"][0], out=state["out"])
    if c["kind"] == "pattern":
        return basis.image_4d(c["half"], c["half"], state["regions"][0], out=state["out"], recompute=True)
    if c["kind"] == "fresh":
        state["spec"].set_atoms(state["atoms"])
        return basis.image(det, state["regions"][0], recompute=True)
    if c["kind"] == "edit":
        spec, images = state["spec"], []
        for (cx, cy), region in zip(state["columns"], state["regions"]):
            spec.edit_column(basis, cx, cy, 0.5, lma.LMA_EDIT_SET_SPECIES, 1)
            images.append(basis.image(det, region))
        for cx, cy in state["columns"]:                        # the next request finds the specimen as it was
            spec.edit_column(basis, cx, cy, 0.5, lma.LMA_EDIT_SET_SPECIES, 0)
        return images
    return basis.image(det, state["regions"][0], out=state["out"], recompute=True)


def work(case):
    """Atoms in, readings out, and the arithmetic of the method: two 2D FFTs, the transmission
    and the propagator per translate and slice, the coefficient products and one 2D FFT per probe."""
    c = case
    W2 = c["window"] ** 2
    slice_flops = W2 * (2 * 5 * math.log2(W2) + 12)
    probe_flops = D * D * (8 * c["L"] + 5 * math.log2(D * D) + 3)
    probes, per_out = c["npx"] * c["npy"], 8 * len(_annuli(c))
    runs, reads = _touched(c) * c["slices"] * c["configs"], probes * c["configs"]
    atoms = 20.0 * 2.5 * c["cells_x"] * c["cells_y"] * c["slices"] * c["configs"]
    store = 4 if c["precision"] == "fp16" else 8
    if c["kind"] == "readout":
        runs = 0
        atoms = float(store) * _touched(c) * W2 * c["configs"]          # resident waves in
    elif c["kind"] == "focal":
        runs, reads = 0, 5 * reads
        atoms = float(store) * _touched(c) * W2 * c["configs"]
    elif c["kind"] == "pattern":
        per_out = 4 * (2 * c["half"] + 1) ** 2
    elif c["kind"] == "edit":
        reach = 2 * R_CUT / WL.ABO3_A * c["nx"] / c["cells_x"] + c["window"]   # windows that meet the column
        near = min(_translates(c), (reach / (c["in_spacing"] * c["f"])) ** 2)
        runs, reads, probes = 2 * near * c["slices"], 2 * reads, 2 * probes
        atoms = 2 * float(store) * _touched(c) * W2
    return {"bytes": atoms + probes * per_out, "flops": runs * slice_flops + reads * probe_flops}


def _touched(c):
    """About how many exit waves the region's probes use."""
    s = c["in_spacing"] * c["f"]
    r = 2.0 * math.sqrt(c["L"] / math.pi) * s
    per = min(c["npx"] * c["npy"] * c["L"],
              (min(c["nx"], c["npx"] * c["spacing_x"] + r) / s) * (min(c["ny"], c["npy"] * c["spacing_y"] + r) / s))
    return max(c["L"], min(_translates(c), per))


# ---------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------
def exact(case, seed):
    c = case
    g, regions = _grid(c), _regions(c, seed)
    need = [_needed(c, r) for r in regions]
    cost = sum(int(n.shape[0]) for n in need) * c["slices"] * c["configs"] * (c["window"] / 128) ** 2.3
    if cost > 2.2e6:
        return None
    atoms = _crystals(c, seed)
    variants = _focal(c) if c["kind"] == "focal" else [(c["defocus"], 0.0, 1.0)]
    images = []
    for k, region in enumerate(regions):
        if c["kind"] == "edit":
            atoms = [_with_column(g, a, _edit_columns(c, seed)[k], 1) for a in atoms]
        total = 0.0
        for a in atoms:
            U = _exit_waves(c, g, a, need[k])
            for defocus, cs, weight in variants:
                total = total + weight * _read(c, g, region, need[k], U, defocus, cs)
            del U
        images.append(total / len(atoms))
    return images if c["kind"] == "edit" else images[0]


def _signed(i, n):
    return i - n if i >= (n + 1) // 2 else i


def _freq(n, d, dev):
    m = torch.tensor([_signed(i, n) for i in range(n)], dtype=torch.float64, device=dev)
    return m, m / (n * d)


def _dev():
    return "cuda:0" if torch.cuda.is_available() else "cpu"


def _probes(c, region):
    b, a = np.meshgrid(np.arange(region.npy), np.arange(region.npx), indexing="ij")
    return ((region.px0 + a * region.spacing_px[0]) % c["nx"]).ravel(), ((region.py0 + b * region.spacing_px[1]) % c["ny"]).ravel()


def _nearest(c, px, py):
    """Offsets (dx, dy) of the L input waves nearest to probe (px, py): by (d^2, dy, dx), periodic."""
    s = c["in_spacing"] * c["f"]
    half = lambda d, n: (d + n // 2) % n - n // 2  # noqa: E731
    dx = half(np.arange(c["in_offset"], c["nx"], s) - px, c["nx"])
    dy = half(np.arange(c["in_offset"], c["ny"], s) - py, c["ny"])
    DY, DX = np.meshgrid(dy, dx, indexing="ij")
    DX, DY = DX.ravel(), DY.ravel()
    order = np.lexsort((DX, DY, DX * DX + DY * DY))[: c["L"]]
    return DX[order], DY[order]


def _classes(c, region):
    """Probes by their place in the input lattice: {class: (probe indices, offsets)}."""
    s = c["in_spacing"] * c["f"]
    px, py = _probes(c, region)
    key = ((px - c["in_offset"]) % s) * s + (py - c["in_offset"]) % s
    out = {}
    for k in np.unique(key):
        at = np.nonzero(key == k)[0]
        out[int(k)] = (at, _nearest(c, px[at[0]], py[at[0]]))
    return out


def _wave_index(c, px, py, dx, dy):
    s = c["in_spacing"] * c["f"]
    ia = ((px + dx - c["in_offset"]) % c["nx"]) // s
    ib = ((py + dy - c["in_offset"]) % c["ny"]) // s
    return ib * (c["nx"] // s) + ia


def _needed(c, region):
    px, py = _probes(c, region)
    mark = np.zeros(_translates(c), bool)
    for at, (dx, dy) in _classes(c, region).values():
        for j in range(len(dx)):
            mark[_wave_index(c, px[at], py[at], dx[j], dy[j])] = True
    return np.nonzero(mark)[0]


def _with_column(g, a, column, species):
    dx, dy = a.x - column[0], a.y - column[1]
    dx, dy = dx - g.lx * np.rint(dx / g.lx), dy - g.ly * np.rint(dy / g.ly)
    sp = a.species.copy()
    sp[dx * dx + dy * dy < 0.25] = species
    return WL.Atoms(a.x, a.y, a.slice, sp)


def _transmissions(g, atoms, dev):
    """exp(i sigma v) per slice: Gaussian sums inside the cutoff, periodic."""
    peak = torch.tensor(PEAKS, dtype=torch.float64, device=dev)
    rx, ry = int(R_CUT / g.dx) + 2, int(R_CUT / g.dy) + 2
    ox = torch.arange(-min(rx, g.nx // 2 - 1), min(rx, g.nx // 2 - 1) + 1, device=dev)
    oy = torch.arange(-min(ry, g.ny // 2 - 1), min(ry, g.ny // 2 - 1) + 1, device=dev)
    for s in range(g.n_slices):
        at = np.nonzero(atoms.slice == s)[0]
        v = torch.zeros(g.ny * g.nx, dtype=torch.float64, device=dev)
        for part in np.array_split(at, max(1, len(at) // 256)):
            x = torch.as_tensor(atoms.x[part], device=dev)
            y = torch.as_tensor(atoms.y[part], device=dev)
            p = peak[torch.as_tensor(atoms.species[part].astype(np.int64), device=dev)]
            ix, iy = torch.round(x / g.dx).long()[:, None] + ox, torch.round(y / g.dy).long()[:, None] + oy
            iyd, ixd = iy.double() * g.dy, ix.double() * g.dx
            r2 = (iyd - y[:, None]).square()[:, :, None] + (ixd - x[:, None]).square()[:, None, :]
            w = sum(f * torch.exp(-r2 / (2 * t * t)) for f, t in zip(TERM_FRAC, TERM_WIDTH)) * p[:, None, None]
            w = torch.where(r2 < R_CUT * R_CUT, w, torch.zeros_like(w))
            v.index_add_(0, ((iy % g.ny)[:, :, None] * g.nx + (ix % g.nx)[:, None, :]).reshape(-1), w.reshape(-1))
        yield torch.polar(torch.ones_like(v), g.sigma * v).reshape(g.ny, g.nx)


def _band(n, frac, dev):
    m = torch.tensor([_signed(i, n) for i in range(n)], dtype=torch.float64, device=dev)
    return 4 * (m[:, None].square() + m[None].square()) <= frac * frac * n * n


def _exit_waves(c, g, atoms, need):
    dev, W = _dev(), c["window"]
    s = c["in_spacing"] * c["f"]
    sigma = g.lam / (2 * GAUSS_ALPHA)
    rx = (torch.arange(W, dtype=torch.float64, device=dev) - W // 2) * g.dx
    ry = (torch.arange(W, dtype=torch.float64, device=dev) - W // 2) * g.dy
    u = torch.exp(-(ry.square()[:, None] + rx.square()[None]) / (2 * sigma * sigma)).to(torch.complex128)
    _, kx = _freq(W, g.dx, dev)
    _, ky = _freq(W, g.dy, dev)
    phase = -math.pi * g.lam * g.slice_dz * (ky.square()[:, None] + kx.square()[None])
    prop = torch.polar(_band(W, g.bandlimit_frac, dev).double(), phase)
    n = torch.as_tensor(need, device=dev)
    tx, ty = c["in_offset"] + (n % (g.nx // s)) * s, c["in_offset"] + (n // (g.nx // s)) * s
    U = u.expand(len(need), W, W).clone()
    step = max(1, (1 << 25) // (W * W))
    ar = torch.arange(W, device=dev)
    for t in _transmissions(g, atoms, dev):
        for i in range(0, len(need), step):
            wx, wy = (tx[i:i + step, None] - W // 2 + ar) % g.nx, (ty[i:i + step, None] - W // 2 + ar) % g.ny
            psi = torch.fft.fft2(U[i:i + step] * t[wy[:, :, None], wx[:, None, :]])
            U[i:i + step] = torch.fft.ifft2(psi.mul_(prop))
    return U


def _coefficients(c, g, dx, dy, defocus, cs):
    """Least squares of the probe (at pixel 0) on its L input waves over the periodic grid."""
    dev, W = _dev(), c["window"]
    _, kx = _freq(g.nx, g.dx, dev)
    _, ky = _freq(g.ny, g.dy, dev)
    k2 = ky.square()[:, None] + kx.square()[None]
    chi = 0.5 * math.pi * cs * g.lam ** 3 * k2.square() - math.pi * defocus * g.lam * k2
    psi = torch.fft.ifft2(torch.polar((g.lam * torch.sqrt(k2) < GAUSS_ALPHA).double(), -chi))
    psi = (psi / torch.linalg.vector_norm(psi)).reshape(-1)
    sigma = g.lam / (2 * GAUSS_ALPHA)
    ar = torch.arange(W, device=dev) - W // 2
    gx = torch.exp(-(ar.double() * g.dx).square() / (2 * sigma * sigma))
    gy = torch.exp(-(ar.double() * g.dy).square() / (2 * sigma * sigma))
    u = gy[:, None] * gx[None]
    rows = np.zeros(g.ny * g.nx, bool)
    places = []
    for j in range(c["L"]):
        at = (((int(dy[j]) + ar) % g.ny)[:, None] * g.nx + ((int(dx[j]) + ar) % g.nx)[None]).reshape(-1)
        places.append(at)
        rows[at.cpu().numpy()] = True
    where = torch.full((g.ny * g.nx,), -1, dtype=torch.long, device=dev)
    live = torch.as_tensor(np.nonzero(rows)[0], device=dev)
    where[live] = torch.arange(live.numel(), device=dev)
    A = torch.zeros(live.numel(), c["L"], dtype=torch.float64, device=dev)
    for j, at in enumerate(places):
        A[where[at], j] = u.reshape(-1)
    q, r = np.linalg.qr(A.cpu().numpy())
    return np.linalg.solve(r.astype(np.complex128), q.T @ psi[live].cpu().numpy())


def _read(c, g, region, need, U, defocus, cs):
    """Synthesized probes' readings [annulus][npy][npx] (or patterns [npy][npx][2 half + 1][2 half + 1])."""
    dev, W = _dev(), c["window"]
    at_wave = np.full(_translates(c), -1)
    at_wave[need] = np.arange(len(need))
    mx, kx = _freq(D, g.dx, dev)
    my, ky = _freq(D, g.dy, dev)
    ang = g.lam * torch.sqrt(ky.square()[:, None] + kx.square()[None])
    band = _band(D, g.bandlimit_frac, dev)
    det = [((ang >= r1) & (ang < r2) & band).double() for r1, r2 in _annuli(c)]
    px, py = _probes(c, region)
    half = c.get("half", 0)
    if c["kind"] == "pattern":
        out = torch.zeros(len(px), 2 * half + 1, 2 * half + 1, dtype=torch.float64, device=dev)
    else:
        out = torch.zeros(len(det), len(px), dtype=torch.float64, device=dev)
    cyclic = W == D == c["nx"] == c["ny"]
    for probes, (dx, dy) in _classes(c, region).values():
        alpha = _coefficients(c, g, dx, dy, defocus, cs)
        for part in np.array_split(probes, -(-len(probes) // 512)):
            psi = torch.zeros(len(part), D, D, dtype=torch.complex128, device=dev)
            for j in range(c["L"]):
                i = torch.as_tensor(at_wave[_wave_index(c, px[part], py[part], dx[j], dy[j])], device=dev)
                sx, sy = int(dx[j]) + (D - W) // 2, int(dy[j]) + (D - W) // 2
                if cyclic:
                    psi += complex(alpha[j]) * torch.roll(U[i], (sy, sx), (1, 2))
                    continue
                x0, x1, y0, y1 = max(0, sx), min(D, sx + W), max(0, sy), min(D, sy + W)
                if x1 > x0 and y1 > y0:
                    psi[:, y0:y1, x0:x1] += complex(alpha[j]) * U[i, y0 - sy:y1 - sy, x0 - sx:x1 - sx]
            p = torch.fft.fft2(psi).abs().square() / (D * D)
            w = torch.as_tensor(part, device=dev)
            if c["kind"] == "pattern":
                ix = torch.arange(-half, half + 1, device=dev) % D
                out[w] = (p * band)[:, ix][:, :, ix]
            else:
                for a, m in enumerate(det):
                    out[a, w] = (p * m).sum((1, 2))
    if c["kind"] == "pattern":
        return out.reshape(c["npy"], c["npx"], 2 * half + 1, 2 * half + 1)
    return out.reshape(len(det), c["npy"], c["npx"])

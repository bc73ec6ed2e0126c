"""Surfaces from delay-Doppler maps (the chunked-DFT path of grids with many
nodes, csrc/dg_map.cu): against the CPU oracle at the FP32 bound, and against
the contraction path (an explicit chunk and tile shape) on what both accept.

Every grid here has at least 8192 nodes (the maps' lower limit)."""
import numpy as np
import pytest

import oracle
import sim
from gpu_common import gpu_surface, lag_boundary_mask, package, rel_err, torch_cuda

pytestmark = pytest.mark.gpu
FP32_TOL = 1e-4


def _scene(seed, spacing, n, k=2, fmt="ci16", fs=20e6, grid=(89, 97), **kw):
    return sim.make_scene(seed=seed, fs_hz=fs, n_samples=n, k_steps=k, fmt=fmt, waveform="noise", snr_db=-3.0,
                          grid_n=grid, grid_spacing_m=spacing, bw_hz=0.9 * fs, **kw)


def _against_oracle(s, c, delay=0, acc=0, npts=1500, seed=1):
    idx = np.unique(np.random.default_rng(seed).integers(0, s.G, npts))
    ref = oracle.cost_points(*oracle.scene_args(s), idx=idx, delay_mode=delay, acc_mode=acc)
    ok = ~lag_boundary_mask(s, idx, delay)
    assert rel_err(c.ravel()[idx][ok], ref[ok], 0.01) < FP32_TOL


# spacings from a few lags to about 6000 (every FFT length, one and several
# lag tiles), captures shorter than one block and of odd length
@pytest.mark.parametrize("spacing,n", [(20.0, 700), (200.0, 3001), (1000.0, 9000), (4000.0, 30001), (12000.0, 20000),
                                       (25000.0, 60001), (25000.0, 2500)])
@pytest.mark.parametrize("delay", [0, 1], ids=["integer", "lagrange4"])
def test_map_surface_matches_oracle(spacing, n, delay):
    s = _scene(40, spacing, n)
    g, c = gpu_surface(s, algo="cdft", delay=["integer", "lagrange4"][delay])
    _against_oracle(s, c, delay)
    g.close()


@pytest.mark.parametrize("fmt", ["c64", "ci16", "ci8"])
@pytest.mark.parametrize("contract", ["fp32", "bf16x3", "fp16x3"])
def test_map_formats_and_arithmetics_on_ragged_grids(fmt, contract):
    """A wide and a tall grid (the lookup's warps splitting the snapshots, and
    one with a row per warp), |C| summed; the arithmetic options share one
    evaluation, so their surfaces are equal."""
    for grid in ((3, 2733), (2733, 3), (401, 1601)):
        s = _scene(41, 300.0, 2049, k=9 if grid[0] == 3 else 2, fmt=fmt, fs=12.5e6, grid=grid)
        g, c = gpu_surface(s, algo="cdft", contract=contract, acc="mag")
        _against_oracle(s, c, acc=1)
        g.close()


def test_map_batches_of_snapshots_and_row_shards():
    """A small scratch target splits the snapshots into batches: the running
    sum continues in the surface, bit for bit. Snapshots of different lengths
    and formats share one plan."""
    torch = torch_cuda()
    P = package()
    s = _scene(42, 500.0, 6000, k=7)
    g, a = gpu_surface(s, algo="cdft", contract="fp16x3")
    g.close()
    g, b = gpu_surface(s, algo="cdft", contract="fp16x3", scratch_mib=1)
    g.close()
    assert np.array_equal(a, b)
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft")
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
    short = 1777
    y1 = torch.from_numpy(s.y1[3][:short].astype(np.float32)).cuda()
    y2 = torch.from_numpy(s.y2[3][:short].astype(np.float32)).cuda()
    g.load_capture(3, "c64", y1, y2)
    c = g.cost_surface().double().cpu().numpy().ravel()
    g.close()
    idx = np.unique(np.random.default_rng(2).integers(0, s.G, 500))
    ref = np.zeros(idx.size)
    for k in range(s.k_steps):
        n = short if k == 3 else s.n_samples
        ref += oracle.cost_points(s.grid, s.ephem[k:k + 1], s.fs_hz, s.fc_hz, oracle.iq_to_f64(s.y1[k:k + 1, :n]),
                                  oracle.iq_to_f64(s.y2[k:k + 1, :n]), idx=idx)
    ok = ~lag_boundary_mask(s, idx)
    assert rel_err(c[idx][ok], ref[ok], 0.01) < FP32_TOL
    # a row shard of the same grid
    g, sh = gpu_surface(s, algo="cdft", row0=1, nrows=87)
    g.close()
    assert rel_err(sh.ravel(), a.reshape(89, 97)[1:88].ravel(), 0.01) < 2 * FP32_TOL


@pytest.mark.parametrize("delay", ["integer", "lagrange4"])
def test_map_lags_without_overlap_and_samples_that_are_not_finite(delay):
    """Captures shorter than the grid's lag range: nodes whose lag leaves no
    overlap are exactly zero. A NaN or an infinity in a c64 capture marks
    exactly the nodes whose overlap touches it, as on the contraction path,
    and leaves the others' values alone."""
    torch = torch_cuda()
    P = package()
    s = _scene(43, 25000.0, 1200, k=1, fmt="c64")
    D, _ = oracle.node_geometry(s.grid, s.ephem, s.fs_hz, s.fc_hz)
    assert np.abs(D).max() > 1300 and np.abs(D).min() < 600

    def surface(y1, y2, **kw):
        g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", delay=delay, **kw)
        g.load_captures("c64", torch.from_numpy(y1).cuda(), torch.from_numpy(y2).cuda())
        c = g.cost_surface().cpu().numpy()
        g.close()
        return c

    rows = dict(chunk=64, tiles="rows")
    a, b = surface(s.y1, s.y2), surface(s.y1, s.y2, **rows)
    assert np.array_equal(a == 0, b == 0) and (a == 0).any()
    y1, y2 = s.y1.copy(), s.y2.copy()
    for pos1, pos2, val in ((None, 1100, np.nan), (40, None, np.inf), (1190, 5, -np.inf)):
        z1, z2 = y1.copy(), y2.copy()
        if pos1 is not None:
            z1[0, pos1, 0] = val
        if pos2 is not None:
            z2[0, pos2, 1] = val
        a2, b2 = surface(z1, z2), surface(z1, z2, **rows)
        bad = ~np.isfinite(b2)
        assert bad.any() and not bad.all()
        assert np.array_equal(np.isnan(a2), bad)
        assert rel_err(a2[~bad], b2[~bad], 0.01) < 2 * FP32_TOL


@pytest.mark.parametrize("window", [(10.0, 200.0), (50.0, 4000.0), (100.0, 15000.0)])
@pytest.mark.parametrize("delay", ["integer", "lagrange4"])
def test_refinement_from_a_table_of_few_lags(window, delay):
    """The refinement around a node (a few lags, summed directly) and windows
    too wide for it: its maximum is the oracle's maximum of the same local grid
    within the bound, and the synchronising call equals the captured step."""
    torch = torch_cuda()
    P = package()
    s = _scene(44, 500.0, 7001, k=3, fmt="c64", fs=12.5e6, grid=(91, 93))
    stream = torch.cuda.Stream()
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", contract="fp16x3", delay=delay, stream=stream)
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
    with torch.cuda.stream(stream):
        cost = g.cost_surface()
        fix = g.argmax_refine(cost, *window)
    lg = oracle.refine_grid(s.grid, fix["index"], *window)
    rows = None if lg["nlat"] < 200 else [fix["ri"]]
    mode = 0 if delay == "integer" else 1
    idx = np.unique(np.r_[fix["ri"] * lg["nlon"] + fix["rj"],
                          np.random.default_rng(3).integers(0, lg["nlat"] * lg["nlon"], 800)])
    ref = oracle.cost_points(lg, s.ephem, s.fs_hz, s.fc_hz, oracle.iq_to_f64(s.y1), oracle.iq_to_f64(s.y2), idx=idx,
                             delay_mode=mode)
    at = ref[np.searchsorted(idx, fix["ri"] * lg["nlon"] + fix["rj"])]
    assert rows is None or fix["refine_n"] == lg["nlat"]
    assert abs(fix["refined_cost"] - at) <= FP32_TOL * at
    assert at >= ref.max() * (1 - 2 * FP32_TOL)
    c2 = torch.empty_like(cost)
    g.graph_capture(c2, *window)
    g.graph_launch()
    assert g.graph_fix() == fix
    g.close()


def test_regions_searched_together_match_fresh_contexts():
    """Regions of many nodes share their launches: every region's surface is
    a fresh context's within twice the bound, the fix its own maximum's."""
    torch = torch_cuda()
    P = package()
    s = _scene(45, 400.0, 6001, k=3, fs=12.5e6, grid=(95, 91))
    offs = [(0.0, 0.0), (0.4, -0.3), (-1.1, 0.8), (2.0, 2.0), (0.05, 0.02)]
    regions = [dict(s.grid, lat0_deg=s.grid["lat0_deg"] + a, lon0_deg=s.grid["lon0_deg"] + b) for a, b in offs]
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", contract="bf16x3")
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
    before = g.cost_surface().clone()
    fix, best, costs = g.search_regions(regions, 20.0, 300.0)
    vals = []
    for r, reg in enumerate(regions):
        f = P.Geolocator(reg, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", contract="bf16x3")
        f.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
        c = f.cost_surface()
        assert rel_err(costs[r].cpu().numpy(), c.cpu().numpy(), 0.01) < 2 * FP32_TOL
        vals.append(float(c.max()))
        f.close()
    assert best == int(np.argmax(vals)) and fix["cost"] == float(costs[best].max())
    assert g.grid["lat0_deg"] == regions[best]["lat0_deg"]
    lo, hi = g.cdft_chunks()
    assert 64 <= lo <= hi <= 2048
    g.set_grid(s.grid)  # the context goes on on its own grid
    assert torch.equal(g.cost_surface(), before)
    g.close()


def test_regions_that_go_around_the_earth():
    """Regions whose first, middle and last columns coincide (two turns): three
    columns bound nothing there, and the regions are searched as fresh contexts."""
    torch = torch_cuda()
    P = package()
    spacing = 4.0 * np.pi * sim.WGS84_A / 2730
    s = sim.make_scene(seed=46, fs_hz=12.5e6, n_samples=4096, k_steps=2, fmt="ci16", waveform="noise", snr_db=-3.0,
                       grid_n=(3, 2731), grid_spacing_m=spacing, bw_hz=10e6, emitter=(0.0, 30.0))
    regions = [dict(s.grid, lon0_deg=s.grid["lon0_deg"] + d) for d in (0.0, 1.0)]
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", contract="fp16x3")
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
    _, _, costs = g.search_regions(regions, 100.0, 1000.0)
    for reg, c in zip(regions, costs.double().cpu().numpy()):
        idx = np.unique(np.random.default_rng(5).integers(0, s.G, 700))
        ref = oracle.cost_points(reg, s.ephem, s.fs_hz, s.fc_hz, oracle.iq_to_f64(s.y1), oracle.iq_to_f64(s.y2), idx=idx)
        ok = ~lag_boundary_mask(s, idx) if reg is regions[0] else np.ones(idx.size, bool)
        D = oracle.node_geometry(reg, s.ephem, s.fs_hz, s.fc_hz)[0].reshape(s.k_steps, -1)[:, idx]
        ok &= (np.abs(D - np.floor(D) - 0.5) > 1e-6).all(axis=0)
        assert rel_err(c.ravel()[idx][ok], ref[ok], 0.01) < FP32_TOL
    g.close()


@pytest.mark.parametrize("delay", [0, 1], ids=["integer", "lagrange4"])
def test_tables_of_thousands_of_bins(delay):
    """A long capture of a wide footprint (more than 2000 Doppler bins, geometry
    per node): away from the peak, where |C| changes with the phase of every sample,
    the 2-norm error stays at the bound of the bins' interpolation (8.4e-7 of the
    coherent sum) and FP32 sums (about as much), twice that in |C|^2; bin
    coordinates rounded to FP32 are off by 1.7e-5 there."""
    s = sim.make_scene(seed=47, fs_hz=1e6, n_samples=131072, k_steps=1, fmt="c64", waveform="noise", snr_db=-3.0,
                       grid_n=(91, 93), grid_spacing_m=9000.0, bw_hz=8e5)
    _, nu = oracle.node_geometry(s.grid, s.ephem, s.fs_hz, s.fc_hz)
    assert np.ptp(nu) * s.n_samples / 7.5e-2 > 2000
    g, c = gpu_surface(s, algo="cdft", delay=["integer", "lagrange4"][delay])
    g.close()
    idx = np.unique(np.random.default_rng(6).integers(0, s.G, 1000))
    ref = oracle.cost_points(*oracle.scene_args(s), idx=idx, delay_mode=delay)
    ok = ~lag_boundary_mask(s, idx, delay)
    ok &= ref < 10 * np.median(ref)
    assert ok.sum() > 900
    assert np.linalg.norm(c.ravel()[idx][ok] - ref[ok]) < 4e-6 * np.linalg.norm(ref[ok])


@pytest.mark.parametrize("fmt,amp", [("ci16", 30000.0), ("c64", 3e5)])
def test_captures_with_pulses(fmt, amp):
    """Isolated pulses hundreds and thousands of times the noise, in both captures:
    an FFT's rounding is relative to the energy of its block, and the surface stays
    within the FP32 bound."""
    torch = torch_cuda()
    P = package()
    s = _scene(48, 200.0, 20000, k=1, fs=12.5e6, grid=(91, 93))
    rng = np.random.default_rng(7)
    y = [rng.normal(0.0, 50.0, (1, 20000, 2)) for _ in range(2)]
    for q in y:
        q[0, rng.integers(0, 20000, 20)] = amp
    y = [np.rint(q).astype(np.int16 if fmt == "ci16" else np.float32) for q in y]
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft")
    g.load_captures(fmt, torch.from_numpy(y[0]).cuda(), torch.from_numpy(y[1]).cuda())
    c = g.cost_surface().double().cpu().numpy().ravel()
    g.close()
    idx = np.unique(rng.integers(0, s.G, 1200))
    ref = oracle.cost_points(s.grid, s.ephem, s.fs_hz, s.fc_hz, oracle.iq_to_f64(y[0]), oracle.iq_to_f64(y[1]), idx=idx)
    ok = ~lag_boundary_mask(s, idx)
    assert rel_err(c[idx][ok], ref[ok], 0.01) < FP32_TOL

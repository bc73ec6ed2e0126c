"""The direct FP32 correlation with the candidates grouped by lag: against
the oracle over group sizes (under and over a warp's 32 and 64 candidates),
both lag sorts, segments of samples that do not divide the capture, formats,
and captures of different lengths in one launch."""
import numpy as np
import pytest

import oracle
import sim
from gpu_common import gpu_surface, lag_boundary_mask, package, rel_err, torch_cuda

pytestmark = pytest.mark.gpu
FP32_TOL = 1e-4


def _check(s, c, acc=0, npts=1200):
    idx = np.unique(np.random.default_rng(1).integers(0, s.G, npts))
    ref = oracle.cost_points(*oracle.scene_args(s), idx=idx, acc_mode=acc)
    ok = ~lag_boundary_mask(s, idx)
    assert rel_err(c.ravel()[idx][ok], ref[ok], 0.01) < FP32_TOL


# (grid, spacing): one lag for many candidates, a few per lag, hundreds per
# lag; grids below and above the one-launch sort's 32768 nodes
@pytest.mark.parametrize("grid,spacing", [((33, 31), 5.0), ((41, 37), 2000.0), ((5, 3000), 100.0), ((190, 181), 150.0)])
@pytest.mark.parametrize("n", [1, 255, 256, 1025, 7003])
def test_lag_groups_match_oracle(grid, spacing, n):
    s = sim.make_scene(seed=61, fs_hz=12.5e6, n_samples=n, k_steps=2, fmt="ci16", waveform="noise", snr_db=-3.0,
                       grid_n=grid, grid_spacing_m=spacing, bw_hz=10e6)
    g, c = gpu_surface(s)
    _check(s, c)
    g.close()


@pytest.mark.parametrize("fmt", ["c64", "ci8"])
def test_lag_groups_of_uneven_captures(fmt):
    """Snapshots of other lengths than the longest (empty last segments) and of
    another format in the same launch."""
    torch = torch_cuda()
    P = package()
    s = sim.make_scene(seed=62, fs_hz=12.5e6, n_samples=5000, k_steps=3, fmt="ci16", waveform="noise", snr_db=-3.0,
                       grid_n=(61, 67), grid_spacing_m=300.0, bw_hz=10e6)
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, acc="mag")
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda())
    n = 300
    dt = np.float32 if fmt == "c64" else np.int8
    a, b = ((y[1][:n] / 100.0).astype(dt) for y in (s.y1, s.y2))
    g.load_capture(1, fmt, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    c = g.cost_surface().double().cpu().numpy().ravel()
    g.close()
    idx = np.unique(np.random.default_rng(2).integers(0, s.G, 600))
    ref = np.zeros(idx.size)
    for k in range(3):
        y1, y2 = (a[None], b[None]) if k == 1 else (s.y1[k:k + 1], s.y2[k:k + 1])
        ref += oracle.cost_points(s.grid, s.ephem[k:k + 1], s.fs_hz, s.fc_hz, oracle.iq_to_f64(y1), oracle.iq_to_f64(y2),
                                  idx=idx, acc_mode=1)
    ok = ~lag_boundary_mask(s, idx)
    assert rel_err(c[idx][ok], ref[ok], 0.01) < FP32_TOL


def _launches(g):
    P = package()
    n0 = P.lib().dg_launch_count(g.ctx)
    g.cost_surface()
    return P.lib().dg_launch_count(g.ctx) - n0


@pytest.mark.parametrize("acc", [0, 1], ids=["power", "mag"])
def test_sparse_lags_keep_the_tile_kernel(acc):
    """Where few candidates share a lag the tile kernel (and the sum over the
    snapshots) runs: its rows per thread change no bit, a row shard is the whole
    grid's rows, and the surface is the oracle's. The same grid on a short baseline
    is grouped by lag."""
    torch = torch_cuda()
    kw = dict(seed=63, fs_hz=60e6, n_samples=50001, k_steps=8, fmt="ci8", waveform="noise", snr_db=-3.0, grid_n=201,
              grid_spacing_m=2000.0, bw_hz=40e6)
    s = sim.make_scene(formation=sim.Formation(sep_m=200e3), **kw)
    D = oracle.node_geometry(s.grid, s.ephem, s.fs_hz, s.fc_hz)[0]
    assert np.abs(D).min() < 45000 and s.G / np.ptp(D[0]) < 3.0
    opts = dict(acc=["power", "mag"][acc])
    g, c = gpu_surface(s, **opts)
    assert _launches(g) == 2
    g.close()
    _check(s, c, acc, 150)
    for rows in (4, 16):
        h, x = gpu_surface(s, rows=rows, **opts)
        assert _launches(h) == 2
        h.close()
        assert np.array_equal(x, c)
    h, x = gpu_surface(s, row0=50, nrows=70, **opts)
    assert _launches(h) == 2
    h.close()
    assert np.array_equal(x, c[50:120])
    near = sim.make_scene(formation=sim.Formation(sep_m=10e3), **kw)
    g, _ = gpu_surface(near, **opts)
    assert _launches(g) > 2
    g.close()


def test_lag_groups_in_batches_of_snapshots():
    """A small scratch target sorts one or two snapshots at a time, and a smaller
    one takes the tile kernel: the grouped surfaces are equal bit for bit."""
    s = sim.make_scene(seed=64, fs_hz=12.5e6, n_samples=3000, k_steps=5, fmt="ci16", waveform="noise", snr_db=-3.0,
                       grid_n=(190, 181), grid_spacing_m=150.0, bw_hz=10e6)
    surfs, launches = [], []
    for mib in (0, 6, 4, 1):
        g, c = gpu_surface(s, scratch_mib=mib)
        surfs.append(c)
        launches.append(_launches(g))
        g.close()
    assert launches[0] < launches[1] < launches[2] and launches[3] == 2
    assert np.array_equal(surfs[1], surfs[0]) and np.array_equal(surfs[2], surfs[0])
    _check(s, surfs[0])
    _check(s, surfs[3])


@pytest.mark.parametrize("lat,grid,turns", [(78.0, (1, 301), 2.0), (84.0, (3, 257), 1.0), (85.5, (61, 67), 0.9)])
def test_lag_slots_of_grids_around_a_pole(lat, grid, turns):
    """Grids whose longitudes go around the Earth once or twice, so that their
    corners and edge midpoints lie close together, and one over the pole."""
    la = np.radians(lat)
    radius = sim.WGS84_A / np.sqrt(1.0 - sim.WGS84_E2 * np.sin(la) ** 2) * np.cos(la)
    spacing = turns * 2.0 * np.pi * radius / (grid[1] - 1)
    s = sim.make_scene(seed=65, fs_hz=12.5e6, n_samples=4096, k_steps=2, fmt="ci16", waveform="noise", snr_db=-3.0,
                       grid_n=grid, grid_spacing_m=spacing, bw_hz=10e6, emitter=(lat, 30.0))
    g, c = gpu_surface(s)
    assert _launches(g) > 2
    fix = g.argmax_refine(g.cost_surface(), 100.0, 1000.0)
    assert fix["refine_n"] == 21
    g.close()
    _check(s, c)


@pytest.mark.parametrize("spacing", [2500.0, 4000.0, 7000.0, 12000.0, 20000.0])
def test_rows_do_not_choose_the_kernel(spacing):
    """Grids on both sides of the rule: one surface for every dg_options.rows."""
    s = sim.make_scene(formation=sim.Formation(sep_m=200e3), seed=66, fs_hz=60e6, n_samples=3000, k_steps=8, fmt="ci8",
                       waveform="noise", snr_db=-3.0, grid_n=101, grid_spacing_m=spacing, bw_hz=40e6)
    surfs, launches = [], []
    for rows in (0, 4, 8, 16):
        g, c = gpu_surface(s, rows=rows)
        surfs.append(c)
        launches.append(_launches(g))
        g.close()
    assert len(set(launches)) == 1
    assert all(np.array_equal(c, surfs[0]) for c in surfs[1:])


def test_sparse_lags_in_a_batch():
    """Small sparse grids group their lags alone, where their tiles leave most SMs
    idle, and keep the tiles in a batch that fills the GPU; the contexts' own calls
    follow the batch while it lives."""
    torch = torch_cuda()
    P = package()
    gs, costs, alone = [], [], []
    for i in range(40):
        s = sim.make_scene(seed=70 + i % 4, fs_hz=20e6, n_samples=2048, k_steps=4, fmt="ci8", waveform="noise", snr_db=-3.0,
                           grid_n=(101, 103), grid_spacing_m=8000.0, bw_hz=16e6)
        g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, stream=torch.cuda.Stream())
        y1, y2 = torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda()
        torch.cuda.synchronize()
        g.load_captures(s.fmt, y1, y2)
        gs.append(g)
        costs.append(torch.empty((g.nrows, g.nlon), dtype=g.dtype, device=g.device))

    def own(g):
        with torch.cuda.stream(g.stream):
            n = _launches(g)
            c = g.cost_surface()
            fix = g.argmax_refine(c, 100.0, 1000.0)
        return n, fix, c.double().cpu().numpy()

    torch.cuda.synchronize()
    alone = [own(g) for g in gs[:4]]
    assert all(n > 2 for n, _, _ in alone)
    b = P.Batch(gs, costs, 100.0, 1000.0)
    b.launch()
    fixes = b.fixes()
    for i in range(4):
        n, fix, c = own(gs[i])
        assert n == 2 and fix == fixes[i]
        assert np.array_equal(costs[i].double().cpu().numpy(), c)
        assert rel_err(c, alone[i][2], 0.01) < 2 * FP32_TOL
    b.close()
    n, fix, c = own(gs[0])
    assert n == alone[0][0] and fix == alone[0][1] and np.array_equal(c, alone[0][2])
    for g in gs:
        g.close()

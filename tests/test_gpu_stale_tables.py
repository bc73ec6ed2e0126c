"""A region search that fails after it has replaced the context's delay-Doppler
tables: a step or batch captured before may not replay on the regions' tables."""
import numpy as np
import pytest

import sim
from gpu_common import package, torch_cuda

pytestmark = pytest.mark.gpu
REFINE = (20.0, 200.0)


@pytest.mark.parametrize("spacing", [60.0, 900.0])
def test_failed_region_search_makes_captured_steps_stale(spacing):
    """No region holds a finite value (a receiver that delivered NaN); with good
    captures again the graph and the batch are refused, as after any other change
    of the context's grid, and a new capture gives the synchronising step's fix."""
    torch = torch_cuda()
    P = package()
    s = sim.make_scene(seed=71, fs_hz=12.5e6, n_samples=9000, k_steps=3, fmt="c64", waveform="noise", snr_db=-3.0,
                       grid_n=(121, 131), grid_spacing_m=200.0, bw_hz=10e6)
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz, algo="cdft", contract="fp16x3", stream=torch.cuda.Stream())
    y1, y2 = torch.from_numpy(s.y1).cuda(), torch.from_numpy(s.y2).cuda()
    torch.cuda.synchronize()
    g.load_captures("c64", y1, y2)
    cost, other = (torch.empty((g.nrows, g.nlon), dtype=g.dtype, device=g.device) for _ in range(2))
    g.graph_capture(cost, *REFINE)
    b = P.Batch([g], [other], *REFINE)
    g.graph_launch()
    ref = g.graph_fix()
    b.launch()
    assert b.fixes() == [ref]
    torch.cuda.synchronize()
    surface = cost.clone()

    bad = torch.full_like(y1, float("nan"))
    torch.cuda.synchronize()
    g.load_captures("c64", bad, y2)
    # regions of another shape than the main grid's, of at least 8192 nodes
    regions = [dict(s.grid, lat0_deg=s.grid["lat0_deg"] + d, nlat=101, nlon=101, dlat_m=spacing, dlon_m=spacing)
               for d in (0.0, 0.3, -0.4)]
    with pytest.raises(P.DGError) as e:
        g.search_regions(regions, *REFINE)
    assert e.value.status == P.DG_EINVAL

    g.load_captures("c64", y1, y2)
    with pytest.raises(P.DGError) as e:
        g.graph_launch()
    assert e.value.status == P.DG_ESTATE
    with pytest.raises(P.DGError) as e:
        b.launch()
    assert e.value.status == P.DG_ESTATE
    with torch.cuda.stream(g.stream):
        assert torch.equal(g.cost_surface(), surface)
    g.graph_capture(cost, *REFINE)
    g.graph_launch()
    assert g.graph_fix() == ref
    torch.cuda.synchronize()
    assert torch.equal(cost, surface)
    b.close()
    g.close()

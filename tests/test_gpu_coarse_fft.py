"""The coarse maps' chunk sums through FFT correlations, the folded chunk DFT and
the pooled back-projection, at the edges of their tiles, against the FP64 oracle.

Tolerances as in test_gpu_coarse.py: 1e-4 (A + mu) per entry of the map (an FP32
transform of n points is off by a few 1e-7 of its root mean square, and the sums
over chunks and |.|^2 add a few 1e-6), and the same per cell where both sides must
take the same box."""
import numpy as np
import pytest

from gpu_common import package, torch_cuda
from oracle import coarse as ocoarse
from test_gpu_coarse import _run, _scene, _unambiguous

pytestmark = pytest.mark.gpu

CASES = [
    # seed, nodes, spacing m, K, N, format, bins, chunk, fs
    (31, (7, 9), 2500.0, 2, 1000, "c64", 17, 128, 5e6),        # middle bin and middle chunk, ragged end
    (32, (5, 6), 3000.0, 1, 1025, "ci16", 256, 1024, 5e6),     # one sample in the last chunk, most bins
    (33, (9, 8), 4000.0, 3, 5000, "ci8", 66, 4096, 5e6),       # longest chunk; bin pairs past two warps
    (34, (33, 35), 30000.0, 2, 2048, "c64", 33, 256, 20e6),    # several lag tiles and boxes of many lags
    (35, (4, 131), 9000.0, 2, 3000, "ci16", 2, 512, 20e6),     # rows longer than a CTA, two bins
    (36, (3, 3), 1000.0, 1, 100, "c64", 8, 512, 5e6),          # a capture shorter than its chunk
]


@pytest.mark.parametrize("case", CASES, ids=[f"seed{c[0]}" for c in CASES])
def test_maps_at_the_edges_of_the_tiles(case):
    seed, nodes, spacing, K, N, fmt, bins, chunk, fs = case
    s = _scene(seed, nodes, spacing, K, N, fmt, fs=fs)
    maps, A, steps, (Q, M, cap) = _run(s, bins, chunk)
    assert (Q, M) == (bins, chunk)
    ref_maps, extra = ocoarse.coarse_maps(s.grid, s.ephem, s.fs_hz, s.fc_hz, s.y1, s.y2, Q, M, want_caf=True)
    for k in range(K):
        (l0, nlag, _, _, _), RA, mu = extra[k]
        assert (steps[k]["l0"], steps[k]["nlag"]) == (l0, nlag)
        assert np.all(np.abs(A[k, :nlag] - RA) <= 1e-4 * (RA + mu)), f"snapshot {k}"
    ok = _unambiguous(s, Q)
    err = np.abs(maps - ref_maps) / (ref_maps + 1.0)
    assert err[ok].max() <= 1e-4


@pytest.mark.parametrize("chunk", [64, 256])  # direct sums, transforms
def test_a_sample_that_is_not_finite_marks_the_lags_that_read_it(chunk):
    torch = torch_cuda()
    P = package()
    s = _scene(37, (21, 21), 3000.0, 2, 4096, "c64")
    y2 = s.y2.copy()
    y2[1, 5, 0] = np.inf  # read by lags up to 5
    g = P.Geolocator(s.grid, s.ephem, s.fs_hz, s.fc_hz)
    g.load_captures(s.fmt, torch.from_numpy(s.y1).cuda(), torch.from_numpy(y2).cuda())
    maps = g.coarse_maps(bins=16, chunk=chunk).cpu().numpy()
    A, steps, _ = g.coarse_inspect()
    A = A.cpu().numpy()
    lags = steps[1]["l0"] + np.arange(steps[1]["nlag"])
    assert np.array_equal(np.isnan(A[1, :lags.size]).all(axis=1), lags <= 5)
    assert np.array_equal(np.isnan(A[1, :lags.size]).any(axis=1), lags <= 5)
    assert np.isfinite(A[0, :steps[0]["nlag"]]).all()
    if (lags <= 5).any():
        assert np.isnan(steps[1]["mu"]) and not maps[1].any()
    y1 = s.y1.copy()
    y1[0, 4000, 1] = np.nan  # every lag's sum
    g.load_captures(s.fmt, torch.from_numpy(y1).cuda(), torch.from_numpy(s.y2).cuda())
    maps = g.coarse_maps(bins=16, chunk=chunk).cpu().numpy()
    A, steps, _ = g.coarse_inspect()
    assert np.isnan(A.cpu().numpy()[0, :steps[0]["nlag"]]).all() and not maps[0].any() and maps[1].any()
    g.close()

"""Performance cases: the calls a user of the library makes, over their range of sizes.

Every case goes through the package's public entry points (``Geolocator``,
``Batch``, ``ProposalNet`` and the layer calls). Inputs are synthetic captures of
one emitter seen by two receivers on one low orbit, made on the GPU from the
seed: the signal differs between the receivers by the delay and the Doppler of
the geometry, with receiver noise, quantised as the capture format asks.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2508_06672_gb300 as P
from paper_2508_06672_gb300.proposal import ProposalNet

DEV = "cuda"
C_LIGHT, FC = 299792458.0, 1575.42e6
WGS_A, WGS_F = 6378137.0, 1.0 / 298.257223563
WGS_E2 = WGS_F * (2.0 - WGS_F)
GM, OMEGA = 3.986004418e14, 7.2921150e-5
BYTES = {"c64": 8, "ci16": 4, "ci8": 2}
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "weights", "proposal_2000km.npz")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: one short capture on a small grid, the default (direct) evaluation; launches count
        dict(name="direct_tiny", kind="surface", nlat=101, nlon=101, spacing=1000.0, K=1, N=4096, fmt="c64",
             fs=5e6, bw=2e6, snr=-5.0, algo="direct", contract="fp32", delay="integer", acc="power"),
        # the plain sample-by-sample search of a survey area, every default option
        dict(name="direct_survey", kind="surface", nlat=301, nlon=403, spacing=300.0, K=4, N=32768, fmt="ci16",
             fs=12.5e6, bw=10e6, snr=-10.0, algo="direct", contract="fp32", delay="integer", acc="power"),
        # one streaming step on a local area: new captures in, surface, argmax and refinement out, synchronising
        dict(name="local_step", kind="step", nlat=121, nlon=131, spacing=200.0, K=4, N=20000, fmt="ci8",
             fs=12.5e6, bw=10e6, snr=-5.0, algo="cdft", contract="fp16x3", delay="integer", acc="power"),
        # the 1001 x 1001 workload with the paper's sum of magnitudes: a whole step replayed as a CUDA graph
        dict(name="mid_graph", kind="graph", nlat=1001, nlon=1001, spacing=100.0, K=20, N=65536, fmt="ci16",
             fs=12.5e6, bw=10e6, snr=-15.0, algo="cdft", contract="fp16x3", delay="integer", acc="mag"),
        # the largest workload: 4001 x 4001 nodes, 50 long captures
        dict(name="large_surface", kind="surface", nlat=4001, nlon=4001, spacing=400.0, K=50, N=131072, fmt="ci8",
             fs=20e6, bw=18e6, snr=-20.0, algo="cdft", contract="fp16x3", delay="integer", acc="power"),
        # fractional delay and magnitudes on a ragged grid and an odd capture length
        dict(name="lagrange_ragged", kind="surface", nlat=263, nlon=397, spacing=500.0, K=6, N=50001, fmt="c64",
             fs=12.5e6, bw=5e6, snr=-10.0, algo="cdft", contract="bf16x3", delay="lagrange4", acc="mag"),
        # the chunked-DFT path with its default arithmetic (FP32)
        dict(name="cdft_default", kind="surface", nlat=257, nlon=257, spacing=400.0, K=8, N=30000, fmt="ci8",
             fs=20e6, bw=18e6, snr=-10.0, algo="cdft", contract="fp32", delay="integer", acc="power"),
        # many uneven captures as one graph
        dict(name="batch_uneven", kind="batch", sides="257,512,301,701,384,997", spacings="400,150,50,250,500,100",
             Ks="5,20,40,10,8,12", Ns="65536,8192,4096,32768,131072,20000", fmt="ci16", fs=12.5e6, bw=10e6, snr=-8.0,
             contract="fp16x3"),
        # the dense stage of the learned search: eight 50 km regions, then the re-evaluation of the best
        dict(name="regions", kind="regions", nreg=8, side=101, spacing=500.0, K=20, N=65536, fmt="ci16", fs=12.5e6,
             bw=10e6, snr=-15.0, contract="bf16x3"),
        # the proposal's coarse delay-Doppler maps over a 2000 km footprint
        dict(name="coarse_maps", kind="coarse", cells=512, footprint=2.0e6, K=20, N=65536, fmt="ci16", fs=12.5e6,
             bw=10e6, snr=-15.0),
        # the shipped proposal network on one footprint's maps (a whole call, its logits)
        dict(name="proposal_forward", kind="forward", cells=512, B=1),
        # training: one layer's gradients at the training batch's shape
        dict(name="conv_backward", kind="convbwd", B=16, Ci=64, Co=128, H=128, W=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["direct", "cdft", "cdft", "cdft", "step", "graph", "batch", "regions", "coarse", "forward",
                       "convbwd"])
    fs = rng.choice([5e6, 12.5e6, 20e6])
    common = dict(fmt=rng.choice(["c64", "ci16", "ci8"]), fs=fs, bw=fs * rng.uniform(0.3, 0.9),
                  snr=round(rng.uniform(-20.0, 0.0), 1))
    if kind == "direct":
        while True:
            c = dict(nlat=_log(rng, 40, 500), nlon=_log(rng, 40, 500), K=rng.randint(1, 8), N=_log(rng, 1000, 60000))
            if c["nlat"] * c["nlon"] * c["K"] * c["N"] < 3e10:
                break
        return dict(kind="surface", spacing=float(_log(rng, 50, 1000)), algo="direct", contract="fp32",
                    delay=rng.choice(["integer", "integer", "lagrange4"]), acc=rng.choice(["power", "mag"]), **c,
                    **common)
    if kind in ("cdft", "step", "graph"):
        contract = rng.choice(["fp16x3", "fp16x3", "bf16x3", "fp32"])
        top, work = (2400, 1.2e13) if contract != "fp32" else (700, 4e11)
        while True:
            c = dict(nlat=_log(rng, 91, top), nlon=_log(rng, 91, top), K=rng.randint(1, 40), N=_log(rng, 4096, 262144))
            if c["nlat"] * c["nlon"] * c["K"] * c["N"] < work and c["K"] * c["N"] < 4e6:
                break
        # short captures sum powers or magnitudes, long ones the paper's magnitudes
        return dict(kind="surface" if kind == "cdft" else kind, spacing=float(_log(rng, 50, 1000)), algo="cdft",
                    contract=contract, delay=rng.choice(["integer", "integer", "integer", "lagrange4"]),
                    acc=rng.choice(["power", "mag"]) if c["K"] * c["N"] < 2e5 else "mag", **c, **common)
    if kind == "batch":
        n = rng.randint(3, 8)
        sides = [_log(rng, 129, 1100) for _ in range(n)]
        Ks = [rng.randint(3, 20) for _ in range(n)]
        Ns = [_log(rng, 4096, 100000) for _ in range(n)]
        return dict(kind="batch", sides=",".join(map(str, sides)),
                    spacings=",".join(str(rng.randint(50, 500)) for _ in range(n)), Ks=",".join(map(str, Ks)),
                    Ns=",".join(map(str, Ns)), contract="fp16x3", **common)
    if kind == "regions":
        K = rng.randint(5, 25)
        return dict(kind="regions", nreg=rng.randint(2, 12), side=rng.randint(45, 70) * 2 + 1,
                    spacing=float(_log(rng, 100, 600)), K=K, N=_log(rng, 8192, 800000 // K),
                    contract=rng.choice(["bf16x3", "fp16x3"]), **common)
    if kind == "coarse":
        return dict(kind="coarse", cells=rng.randint(96, 512), footprint=float(_log(rng, 300000, 2000000)),
                    K=rng.randint(4, 24), N=_log(rng, 8192, 80000), **common)
    if kind == "forward":
        return dict(kind="forward", cells=rng.randint(100, 512), B=rng.randint(1, 2))
    return dict(kind="convbwd", B=rng.randint(1, 16), Ci=rng.choice([20, 32, 64, 96, 128]),
                Co=rng.choice([1, 32, 64, 128]), H=rng.randint(40, 160), W=rng.randint(40, 160))


# ------------------------------------------------------------------- inputs
def _ecef(lat_deg, lon_deg):
    la, lo = math.radians(lat_deg), math.radians(lon_deg)
    n = WGS_A / math.sqrt(1.0 - WGS_E2 * math.sin(la) ** 2)
    return np.array([n * math.cos(la) * math.cos(lo), n * math.cos(la) * math.sin(lo),
                     n * (1.0 - WGS_E2) * math.sin(la)])


def _state(t, u0):
    """ECEF position and velocity on a circular orbit (550 km, 53 degrees) at argument of latitude u0 at t = 0."""
    r = WGS_A + 550e3
    n = math.sqrt(GM / r ** 3)
    u, inc, th = u0 + n * t, math.radians(53.0), OMEGA * t
    pos = r * np.array([math.cos(u), math.sin(u) * math.cos(inc), math.sin(u) * math.sin(inc)])
    vel = r * n * np.array([-math.sin(u), math.cos(u) * math.cos(inc), math.cos(u) * math.sin(inc)])
    rot = np.array([[math.cos(th), math.sin(th), 0], [-math.sin(th), math.cos(th), 0], [0, 0, 1.0]])
    p = rot @ pos
    return p, rot @ vel - np.cross([0, 0, OMEGA], p)


def _ephem(K, u0):
    """(K, 12) receiver states 1 s apart, receiver 2 leading by 50 km of arc."""
    du = 50e3 / (WGS_A + 550e3)
    return np.array([np.concatenate(_state(k, u0) + _state(k, u0 + du)) for k in range(K)])


def _ground(K, u0, along, cross):
    """The point `along` and `cross` metres from the formation's ground track at mid-time, in degrees."""
    p, v = _state(0.5 * (K - 1), u0)
    g = p / np.linalg.norm(p)
    t = v - (v @ g) * g
    t /= np.linalg.norm(t)
    a, c = along / WGS_A, cross / WGS_A
    e = math.cos(c) * (math.cos(a) * g + math.sin(a) * t) + math.sin(c) * np.cross(g, t)
    return math.degrees(math.asin(e[2])), math.degrees(math.atan2(e[1], e[0]))


def _captures(seed, eph, site, N, fmt, fs, bw, snr):
    """Both receivers' captures, (K, N, 2) on the GPU: band-limited noise from `site`, delayed and Doppler-shifted
    by the geometry, plus receiver noise of unit power."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    pe, K = _ecef(*site), eph.shape[0]
    n_fft = 1 << int(math.ceil(math.log2(2 * N + 8192)))
    f = torch.fft.fftfreq(n_fft, 1.0 / fs, dtype=torch.float64, device=DEV)
    t = torch.arange(N, dtype=torch.float64, device=DEV) / fs
    amp = 10.0 ** (snr / 20.0)
    dtype = {"c64": torch.float32, "ci16": torch.int16, "ci8": torch.int8}[fmt]
    out = [torch.empty((K, N, 2), dtype=dtype, device=DEV) for _ in range(2)]
    std = math.sqrt((amp * amp + 1.0) / 2.0)
    for k in range(K):
        spec = torch.randn(n_fft, dtype=torch.complex64, device=DEV, generator=gen).to(torch.complex128)
        spec = spec * (f.abs() <= 0.5 * bw)
        spec = spec * (n_fft / torch.linalg.vector_norm(spec))
        d0 = None
        for r in range(2):
            p, v = eph[k, 6 * r:6 * r + 3], eph[k, 6 * r + 3:6 * r + 6]
            rng_m = float(np.linalg.norm(p - pe))
            dop = -float((p - pe) @ v) / rng_m * FC / C_LIGHT
            d0 = rng_m / C_LIGHT if d0 is None else d0
            x = torch.fft.ifft(spec * torch.exp(-2j * math.pi * f * (rng_m / C_LIGHT - d0)))[:N]
            x = amp * x * torch.exp(2j * math.pi * dop * t)
            x = x + torch.randn(N, dtype=torch.complex64, device=DEV, generator=gen)
            y = torch.view_as_real(x)
            if fmt == "ci16":
                y = (y * (2048.0 / std)).round().clamp(-32767, 32767)
            elif fmt == "ci8":
                y = (y * (24.0 / std)).round().clamp(-127, 127)
            out[r][k] = y.to(dtype)
    return out


def _grid(site, nlat, nlon, spacing):
    return dict(lat0_deg=site[0], lon0_deg=site[1], dlat_m=spacing, dlon_m=spacing, nlat=nlat, nlon=nlon)


def _scene(case, seed, nlat, nlon, spacing, K, N):
    """A scene whose grid is centred on the emitter, 150 to 450 km beside the ground track."""
    rng = np.random.default_rng(seed)
    u0 = math.radians(20.0)
    site = _ground(K, u0, rng.uniform(-150e3, 150e3), rng.choice([-1.0, 1.0]) * rng.uniform(150e3, 450e3))
    eph = _ephem(K, u0)
    y1, y2 = _captures(seed, eph, site, N, case["fmt"], case["fs"], case["bw"], case["snr"])
    return dict(grid=_grid(site, nlat, nlon, spacing), eph=eph, y1=y1, y2=y2, rng=rng, site=site)


def _locator(case, s, grid=None, stream=None, **kw):
    opts = dict(algo=case.get("algo", "cdft"), contract=case.get("contract", "fp32"),
                delay=case.get("delay", "integer"), acc=case.get("acc", "power"))
    opts.update(kw)
    g = P.Geolocator(grid or s["grid"], s["eph"], case["fs"], FC, stream=stream, **opts)
    g.load_captures(case["fmt"], s["y1"], s["y2"])
    return g


def _ints(text):
    return [int(x) for x in text.split(",")]


def _net_inputs(case, seed):
    """Coarse maps as the library makes them: positive, mean about one per bin before the max-pool, with a ridge."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n, K = case["cells"], 20
    u = torch.rand((case["B"], K, n, n), device=DEV, generator=gen).clamp_min(1e-7)
    maps = -torch.log1p(-u.pow(1.0 / 12.0)).clamp_max(-1e-7)  # the largest of 12 exponentials
    i = torch.arange(n, device=DEV, dtype=torch.float32)
    for k in range(K):
        d = (i[:, None] - 0.4 * n) + (0.2 + 0.01 * k) * (i[None, :] - 0.6 * n)
        maps[:, k] += 6.0 * torch.exp(-0.5 * (d / 1.5) ** 2)
    return maps.contiguous()


def _conv_inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    B, Ci, Co, H, W = (case[k] for k in ("B", "Ci", "Co", "H", "W"))
    x = torch.randn((B, Ci, H, W), device=DEV, generator=gen).clamp_min(0.0)  # activations after a relu
    w = torch.randn((Co, Ci, 3, 3), device=DEV, generator=gen) * math.sqrt(2.0 / (9 * Ci))
    dy = torch.randn((B, Co, H, W), device=DEV, generator=gen) * 1e-4
    return x, w, dy


# -------------------------------------------------------------- the contract
def prepare(case, seed):
    kind = case["kind"]
    if kind == "forward":
        return dict(kind=kind, net=ProposalNet.load(WEIGHTS), x=_net_inputs(case, seed))
    if kind == "convbwd":
        x, w, dy = _conv_inputs(case, seed)
        scratch = torch.empty(int(P.lib().dg_nn_conv3x3_tc_scratch(case["B"], case["Ci"], case["Co"], case["H"],
                                                                   case["W"])), device=DEV)
        return dict(kind=kind, x=x, w=w, dy=dy, dx=torch.empty_like(x), dw=torch.empty_like(w),
                    db=torch.empty(case["Co"], device=DEV), scratch=scratch)
    if kind == "batch":
        gs, costs = [], []
        for j, (side, sp, K, N) in enumerate(zip(*(_ints(case[k]) for k in ("sides", "spacings", "Ks", "Ns")))):
            s = _scene(case, seed * 131 + j, side, side, float(sp), K, N)
            torch.cuda.synchronize()
            gs.append(_locator(case, s, stream=torch.cuda.Stream(), scratch_mib=256))
            costs.append(torch.empty((side, side), device=DEV))
            torch.cuda.synchronize()
        return dict(kind=kind, batch=P.Batch(gs, costs, 10.0, 200.0), gs=gs, costs=costs)
    if kind == "regions":
        s = _scene(case, seed, case["side"], case["side"], case["spacing"], case["K"], case["N"])
        g = _locator(case, s)
        regions = []
        for j in range(case["nreg"]):  # the first holds the emitter, the others lie around it
            off = s["rng"].uniform(-3.0, 3.0, 2) if j else s["rng"].uniform(-0.1, 0.1, 2)
            regions.append(dict(s["grid"], lat0_deg=s["grid"]["lat0_deg"] + off[0],
                                lon0_deg=s["grid"]["lon0_deg"] + off[1]))
        return dict(kind=kind, g=g, regions=regions,
                    costs=torch.empty((case["nreg"], case["side"], case["side"]), device=DEV))
    if kind == "coarse":
        rng = np.random.default_rng(seed)
        u0 = math.radians(86.0)  # near the orbit's northern apex, the footprint on one side of the track
        centre = _ground(case["K"], u0, 0.0, -1.2e6 if _ground(9, u0, 0.0, 1e3)[0] > _ground(9, u0, 0.0, -1e3)[0]
                         else 1.2e6)
        site = (centre[0] + rng.uniform(-1.0, 1.0), centre[1] + rng.uniform(-1.0, 1.0))
        eph = _ephem(case["K"], u0)
        y1, y2 = _captures(seed, eph, site, case["N"], case["fmt"], case["fs"], case["bw"], case["snr"])
        n = case["cells"]
        g = _locator(dict(case, algo="cdft", contract="bf16x3"), dict(eph=eph, y1=y1, y2=y2),
                     grid=_grid(centre, n + 1, n + 1, case["footprint"] / n))
        return dict(kind=kind, g=g, maps=torch.empty((case["K"], n, n), device=DEV))
    s = _scene(case, seed, case["nlat"], case["nlon"], case["spacing"], case["K"], case["N"])
    cost = torch.empty((case["nlat"], case["nlon"]), device=DEV)
    if kind == "graph":
        torch.cuda.synchronize()
        g = _locator(case, s, stream=torch.cuda.Stream())
        g.graph_capture(cost, 10.0, 200.0)
        return dict(kind=kind, g=g, cost=cost)
    return dict(kind=kind, g=_locator(case, s), cost=cost, fmt=case["fmt"], y1=s["y1"], y2=s["y2"])


def _fix(f):
    return torch.tensor([f["cost"], f["refined_cost"]], dtype=torch.float32)


def run(state):
    kind = state["kind"]
    if kind == "surface":
        return state["g"].cost_surface(out=state["cost"])
    if kind == "step":
        g = state["g"]
        g.load_captures(state["fmt"], state["y1"], state["y2"])
        cost = g.cost_surface(out=state["cost"])
        return cost, _fix(g.argmax_refine(cost, 10.0, 200.0))
    if kind == "graph":
        state["g"].graph_launch()
        return state["cost"], _fix(state["g"].graph_fix())
    if kind == "batch":
        state["batch"].launch()
        fixes = state["batch"].fixes()
        return state["costs"] + [_fix(f) for f in fixes]
    if kind == "regions":
        fix, best, costs = state["g"].search_regions(state["regions"], 25.0, 500.0, costs=state["costs"])
        return costs, _fix(fix)
    if kind == "coarse":
        return state["g"].coarse_maps(out=state["maps"])
    if kind == "forward":
        return state["net"].forward(state["x"])
    P.dg_nn_conv3x3_backward_tc(state["x"], state["w"], state["dy"], state["dx"], state["dw"], state["db"],
                                scratch=state["scratch"])
    return state["dx"], state["dw"], state["db"]


def _channels():
    return [20, 32, 64, 128, 64, 1]


def work(case):
    """Captures in, surfaces out. flops of a surface: the 14 of one candidate and sample for the direct evaluation;
    for the chunked-DFT path what a correlation over all lags costs through FFTs is far less, so only the work on
    each candidate and snapshot (geometry and interpolation, about 100) and a pass over the samples are counted."""
    kind = case["kind"]
    if kind == "forward":
        px, ch = case["B"] * case["cells"] ** 2, _channels()
        return dict(bytes=4 * px * (ch[0] + 1), flops=sum(18 * a * b for a, b in zip(ch, ch[1:])) * px)
    if kind == "convbwd":
        px = case["B"] * case["H"] * case["W"]
        return dict(bytes=4 * px * (2 * case["Ci"] + case["Co"]), flops=36 * px * case["Ci"] * case["Co"])
    if kind == "coarse":
        cells = case["K"] * case["cells"] ** 2
        return dict(bytes=2 * BYTES[case["fmt"]] * case["K"] * case["N"] + 4 * cells, flops=100 * cells)
    if kind == "batch":
        z = list(zip(*(_ints(case[k]) for k in ("sides", "Ks", "Ns"))))
        return dict(bytes=sum(2 * BYTES[case["fmt"]] * K * N + 4 * a * a for a, K, N in z),
                    flops=sum(100 * a * a * K + 100 * K * N for a, K, N in z))
    G = case["nreg"] * case["side"] ** 2 if kind == "regions" else case["nlat"] * case["nlon"]
    K, N = case["K"], case["N"]
    direct = case.get("algo") == "direct"
    return dict(bytes=2 * BYTES[case["fmt"]] * K * N + 4 * G, flops=14 * G * K * N if direct else 100 * K * (G + N))


# ------------------------------------------------------------- 64-bit values
def _nodes(grid):
    """ECEF of every node, float64 (3, G)."""
    la0, lo0 = math.radians(grid["lat0_deg"]), math.radians(grid["lon0_deg"])
    w = math.sqrt(1.0 - WGS_E2 * math.sin(la0) ** 2)
    dla = grid["dlat_m"] / (WGS_A * (1.0 - WGS_E2) / w ** 3)
    dlo = grid["dlon_m"] / (WGS_A / w * math.cos(la0))
    i = torch.arange(grid["nlat"], dtype=torch.float64, device=DEV) - 0.5 * (grid["nlat"] - 1)
    j = torch.arange(grid["nlon"], dtype=torch.float64, device=DEV) - 0.5 * (grid["nlon"] - 1)
    la, lo = torch.meshgrid(la0 + i * dla, lo0 + j * dlo, indexing="ij")
    n = WGS_A / torch.sqrt(1.0 - WGS_E2 * torch.sin(la) ** 2)
    return torch.stack([n * torch.cos(la) * torch.cos(lo), n * torch.cos(la) * torch.sin(lo),
                        n * (1.0 - WGS_E2) * torch.sin(la)]).reshape(3, -1)


def _surface64(grid, eph, y1, y2, fs, delay, acc):
    """The correlation of every candidate with every snapshot, summed over samples and snapshots, in 64 bits."""
    xyz = _nodes(grid)
    G, (K, N) = xyz.shape[1], y1.shape[:2]
    M = 256  # e^{j 2 pi nu n} = e^{j 2 pi nu M b} e^{j 2 pi nu m}, n = M b + m: exact, and far fewer exponentials
    nb = -(-N // M)
    total = torch.zeros(G, dtype=torch.float64, device=DEV)
    m = torch.arange(M, dtype=torch.float64, device=DEV)
    b = torch.arange(nb, dtype=torch.float64, device=DEV) * M
    for k in range(K):
        f, r = [], []
        for q in range(2):
            p = torch.tensor(eph[k, 6 * q:6 * q + 3], device=DEV)[:, None] - xyz
            v = torch.tensor(eph[k, 6 * q + 3:6 * q + 6], device=DEV)[:, None]
            r.append(torch.sqrt((p * p).sum(0)))
            f.append(-(p * v).sum(0) / (r[q] * (C_LIGHT / FC)))
        D = (r[1] - r[0]) / C_LIGHT * fs
        nu = (f[1] - f[0]) / fs
        L = torch.floor(D) if delay == "lagrange4" else torch.sign(D) * torch.floor(D.abs() + 0.5)
        mu = D - L
        L = L.long()
        a = torch.view_as_complex(y1[k].double())
        a = torch.cat([a, a.new_zeros(nb * M - N)])
        pad = int(L.abs().max()) + 4
        z2 = torch.view_as_complex(y2[k].double()).conj()
        z2 = torch.cat([z2.new_zeros(pad), z2, z2.new_zeros(nb * M - N + pad)])
        taps = [(0, torch.ones_like(mu))]
        if delay == "lagrange4":
            taps = [(-1, -mu * (mu - 1) * (mu - 2) / 6), (0, (mu + 1) * (mu - 1) * (mu - 2) / 2),
                    (1, -(mu + 1) * mu * (mu - 2) / 2), (2, (mu + 1) * mu * (mu - 1) / 6)]
        windows = z2.unfold(0, nb * M, 1)  # row l + pad: y2 shifted by l
        step = max(1, (1 << 27) // (nb * M))
        for g0 in range(0, G, step):
            sl = slice(g0, g0 + step)
            e1 = torch.polar(torch.ones_like(nu[sl])[:, None].expand(-1, M), 2 * math.pi * nu[sl, None] * m)
            e2 = torch.polar(torch.ones_like(nu[sl])[:, None].expand(-1, nb), 2 * math.pi * nu[sl, None] * b)
            c = 0
            for d, wt in taps:
                z = (windows[L[sl] + d + pad] * a).view(-1, nb, M)
                c = c + wt[sl] * (torch.bmm(z, e1[:, :, None])[:, :, 0] * e2).sum(1)
            pw = c.real ** 2 + c.imag ** 2
            total[sl] += pw if acc == "power" else torch.sqrt(pw)
    return total.view(grid["nlat"], grid["nlon"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "forward":
        h, z = _net_inputs(case, seed).double(), np.load(WEIGHTS)
        n = len(z["channels"]) - 1
        for k in range(n):
            h = torch.nn.functional.conv2d(h, torch.tensor(z[f"w{k}"], device=DEV).double(),
                                           torch.tensor(z[f"b{k}"], device=DEV).double(), padding=1)
            h = torch.relu(h) if k < n - 1 else h
        return h
    if kind == "convbwd":
        x, w, dy = (t.double() for t in _conv_inputs(case, seed))
        dx = torch.nn.functional.conv_transpose2d(dy, w, padding=1)
        H, W = x.shape[2:]
        xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
        dw = torch.stack([torch.stack([torch.einsum("bohw,bchw->oc", dy, xp[:, :, u:u + H, v:v + W])
                                       for v in range(3)], -1) for u in range(3)], -2)
        return dx, dw, dy.sum((0, 2, 3))
    if kind in ("batch", "coarse"):
        return None
    if kind == "regions":
        if case["nreg"] * case["side"] ** 2 * case["K"] * case["N"] > 1.5e11:
            return None
        s = _scene(case, seed, case["side"], case["side"], case["spacing"], case["K"], case["N"])
        out = []
        for j in range(case["nreg"]):
            off = s["rng"].uniform(-3.0, 3.0, 2) if j else s["rng"].uniform(-0.1, 0.1, 2)
            grid = dict(s["grid"], lat0_deg=s["grid"]["lat0_deg"] + off[0], lon0_deg=s["grid"]["lon0_deg"] + off[1])
            out.append(_surface64(grid, s["eph"], s["y1"], s["y2"], case["fs"], "integer", "power"))
        return torch.stack(out), None
    taps = 4 if case["delay"] == "lagrange4" else 1
    if case["nlat"] * case["nlon"] * case["K"] * case["N"] * taps > 1.5e11:
        return None
    s = _scene(case, seed, case["nlat"], case["nlon"], case["spacing"], case["K"], case["N"])
    c = _surface64(s["grid"], s["eph"], s["y1"], s["y2"], case["fs"], case["delay"], case["acc"])
    return c if kind == "surface" else (c, None)

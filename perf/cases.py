"""Timed cases of the SBR channel-modelling library: what its users have it do.

A case is a dict of plain values. `listed` gives the standing set, `draw` one
more case of the same ranges, `prepare` the inputs and handles a program holds
before the call, `run` one pass through the public entry points, `work` the
bytes and operations a pass cannot do without, and `exact` the results in 64-bit
arithmetic by plain numpy and torch where the paths have a closed form.

Kinds of case:
  link       scene to channel: BVH build, trace, paths, gains, PDP (and H for a
             single antenna pair), the pipeline run once per Tx position
  synth      H(f) of one receiver for given paths (FP16x3, BF16x3, FP32, FP64)
  elements   H(f) with every receive element traced as its own receiver
  capacity   MIMO capacity of an H(f) over a list of SNRs
  targets    gains at several frequencies and the surrogate's training targets
  train      one optimiser step of the surrogate network
  predict    the surrogate's answers to a set of queries
  batch      many uneven Tx-Rx jobs over several scenes as one launch

The paths of synth, elements and targets are those of an empty rectangular
room, whose images are known in closed form; they enter the library as trace
records (the form in which traces of ray ranges are merged).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2208_10006_gb300 as sbr

C0 = 299792458.0
EPS0 = 8.8541878128e-12
MATERIALS = ((5.31, 0.5), (6.27, 0.1), (3.0, 0.01))   # eps_r, S/m
PRECISION = {"fp64": sbr.SYNTH_FP64, "fp32": sbr.SYNTH_FP32, "bf16x3": sbr.SYNTH_BF16X3, "fp16x3": sbr.SYNTH_FP16X3}
N_OUT, N_TAPS, TAP_S, FLOOR_DB = 20, 16, 5e-9, -40.0   # surrogate outputs: loss, spread, taps, coverage, error head


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest whole call: a single antenna pair in a street scene at 28 GHz, 100,002 rays; launches and waits count
        dict(name="link_street_siso", kind="link", scene="street", N=100, K=3, n_rx=1, F=1, tri=14, sah=False, pol="V"),
        # an indoor massive-MIMO link: furnished room, 4 M rays, one receiver, 1024 subcarriers
        dict(name="link_room_ofdm", kind="link", scene="room", N=632, K=4, n_rx=1, F=1024, tri=5736, sah=False, pol="V"),
        # coverage of a city district at 300 GHz: 10 M rays, six reflections, 1024 receivers (the benchmark's workload)
        dict(name="link_urban_coverage", kind="link", scene="urban", N=1000, K=6, n_rx=1024, F=1, tri=51600, sah=False, pol="V"),
        # H(f) of a 16 x 16 array to 64 elements over 1024 subcarriers on the tensor cores
        dict(name="synth_fp16x3", kind="synth", precision="fp16x3", F=1024, Nr=64, Nt=256, K=3, pol="V"),
        # the default precision on an odd array: 63 transmit and 13 receive elements, 600 subcarriers, 129 paths
        dict(name="synth_fp32_odd", kind="synth", precision="fp32", F=600, Nr=13, Nt=63, K=4, pol="H"),
        # the 64-bit sum that the other precisions are checked with, at a size used for that
        dict(name="synth_fp64", kind="synth", precision="fp64", F=128, Nr=16, Nt=64, K=3, pol="V"),
        # spatially non-stationary channel: 64 receive elements, each with its own paths
        dict(name="elements_fp32", kind="elements", precision="fp32", F=512, Nr=64, Nt=256, K=3, pol="V"),
        # capacity of the full indoor H at seven SNRs
        dict(name="capacity_64x256", kind="capacity", F=1024, Nr=64, Nt=256, n_snr=7),
        # training data of the surrogate: 4096 receivers x 8 frequencies
        dict(name="targets_4096rx", kind="targets", n_rx=4096, F=8, K=2, pol="V"),
        # one optimiser step at the batch size the surrogate is trained with
        dict(name="train_8192", kind="train", B=8192, width=256, depth=4),
        # a map's worth of queries in one call
        dict(name="predict_1M", kind="predict", B=1048576, width=256, depth=4),
        # uneven Tx-Rx jobs over four districts, 1e5 to 1e7 rays each, as one graph launch
        dict(name="batch_24jobs", kind="batch", jobs=24, scenes=4, n_min=100, n_max=1000, tri=20000, f_max=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["link", "link", "synth", "synth", "elements", "capacity", "targets", "train", "predict", "batch"])
    pol = rng.choice(["V", "H"])
    if kind == "link":
        scene = rng.choice(["street", "room", "urban"])
        urban = scene == "urban"
        return dict(kind=kind, scene=scene, N=_log(rng, 30, 632 if scene == "room" else 1000),
                    K=rng.randint(1, 6 if urban else 4), n_rx=_log(rng, 1, 1024) if urban else 1,
                    F=1 if urban else _log(rng, 1, 1024), tri={"street": 14, "room": 5736, "urban": _log(rng, 1000, 51600)}[scene],
                    sah=rng.random() < 0.25, pol=pol)
    if kind == "synth":
        p = rng.choice(["fp16x3", "fp16x3", "bf16x3", "fp32", "fp32", "fp64"])
        small = p == "fp64"
        return dict(kind=kind, precision=p, F=_log(rng, 1, 128 if small else 1024), Nr=_log(rng, 1, 16 if small else 64),
                    Nt=_log(rng, 1, 64 if small else 256), K=rng.randint(1, 3 if small else 4), pol=pol)
    if kind == "elements":
        return dict(kind=kind, precision="fp32", F=_log(rng, 8, 512), Nr=_log(rng, 2, 64), Nt=_log(rng, 1, 256),
                    K=rng.randint(1, 3), pol=pol)
    if kind == "capacity":
        return dict(kind=kind, F=_log(rng, 16, 1024), Nr=_log(rng, 1, 64), Nt=_log(rng, 1, 256), n_snr=rng.randint(1, 7))
    if kind == "targets":
        return dict(kind=kind, n_rx=_log(rng, 16, 4096), F=rng.randint(1, 8), K=rng.randint(1, 2), pol=pol)
    if kind == "train":
        return dict(kind=kind, B=_log(rng, 256, 8192), width=rng.choice([128, 256]), depth=rng.randint(2, 4))
    if kind == "predict":
        return dict(kind=kind, B=_log(rng, 1, 1048576), width=rng.choice([128, 256]), depth=rng.randint(2, 4))
    return dict(kind=kind, jobs=rng.randint(3, 24), scenes=rng.randint(1, 4), n_min=60, n_max=_log(rng, 120, 900),
                tri=_log(rng, 1000, 20000), f_max=rng.choice([64, 256, 1024]))


# ---------------------------------------------------------------- geometry
def _face(axis, value, u, v):
    """Triangles of an axis-aligned rectangle over the lattices u, v of the other two axes."""
    ua, va = [a for a in range(3) if a != axis]
    q = np.empty((len(u), len(v), 3))
    q[..., axis] = value
    q[..., ua], q[..., va] = u[:, None], v[None, :]
    a, b, c, d = q[:-1, :-1], q[1:, :-1], q[1:, 1:], q[:-1, 1:]
    return np.stack([np.stack([a, b, c], 2), np.stack([a, c, d], 2)], 2).reshape(-1, 3, 3)


def _box(lo, hi, n, faces=6):
    """x-, x+, y-, y+, then z+ (five faces) or z-, z+ (six), each of n x n quads."""
    lat = [np.linspace(lo[a], hi[a], n + 1) for a in range(3)]
    order = [(0, 0), (0, 1), (1, 0), (1, 1)] + ([(2, 0), (2, 1)] if faces == 6 else [(2, 1)])
    return [_face(a, (lo, hi)[s][a], *[lat[k] for k in range(3) if k != a]) for a, s in order]


def _materials(rng, S):
    m = np.empty((S, 3))
    m[:, :2] = np.array(MATERIALS)[rng.integers(0, 3, S)]
    m[:, 2] = rng.uniform(0.05e-3, 0.3e-3, S)
    return m


def _city(rng, nx, ny, sub, ground):
    """nx x ny buildings on a 60 m pitch over a tiled ground."""
    groups = [_face(2, 0.0, np.linspace(-20.0, 60.0 * nx + 20, ground + 1), np.linspace(-20.0, 60.0 * ny + 20, ground + 1))]
    for i in range(nx):
        for j in range(ny):
            w, d, h = rng.uniform(15, 40), rng.uniform(15, 40), rng.uniform(10, 60)
            cx, cy = 30 + 60 * i, 30 + 60 * j
            groups += _box((cx - w / 2, cy - d / 2, 0.0), (cx + w / 2, cy + d / 2, h), sub, faces=5)
    return groups


def _furnished(rng):
    """A 10 x 8 x 3 m room with 46 pieces of furniture away from both arrays."""
    groups = _box((0, 0, 0), (10, 8, 3), 8)
    while len(groups) < 6 * 47:
        sx, sy, h = rng.uniform(0.3, 1.5), rng.uniform(0.3, 1.5), rng.uniform(0.4, 2.0)
        cx, cy = rng.uniform(sx / 2, 10 - sx / 2), rng.uniform(sy / 2, 8 - sy / 2)
        if any(abs(cx - x) < sx / 2 + 0.6 and abs(cy - y) < sy / 2 + 0.6 for x, y in ((0.5, 4.0), (8.5, 3.0))):
            continue
        groups += _box((cx - sx / 2, cy - sy / 2, 0.0), (cx + sx / 2, cy + sy / 2, h), 3)
    return groups


def _dev(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _mesh(groups):
    tri = np.concatenate(groups).reshape(-1, 9)
    sid = np.repeat(np.arange(len(groups)), [len(g) for g in groups])
    return _dev(tri, torch.float32), _dev(sid, torch.int32)


def _grid(fc, F):
    return fc + (np.arange(F) - F // 2) * (min(10e9, fc / 10) / F)


def _upa(center, n, spacing):
    """n elements in the y-z plane, as square as they come."""
    side = max(1, math.isqrt(n))
    k = np.arange(n)
    p = np.tile(np.asarray(center, np.float64), (n, 1))
    p[:, 1] += ((k % side) - (side - 1) / 2) * spacing
    p[:, 2] += ((k // side) - ((n - 1) // side) / 2) * spacing
    return p


def _ula(center, n, spacing):
    p = np.tile(np.asarray(center, np.float64), (n, 1))
    p[:, 1] += (np.arange(n) - (n - 1) / 2) * spacing
    return p


# ---------------------------------------------------------------- the empty room in closed form
ROOM = np.array([10.0, 8.0, 3.0])


def room_paths(tx, rx, K):
    """Specular paths of up to K reflections between tx and each rx in the empty room, by unfolding it:
    receiver, reflections, walls (2 axis + side), points and lengths, in the order (receiver, reflections, walls)."""
    I = np.array([(i, j, k) for i in range(-K, K + 1) for j in range(-K, K + 1) for k in range(-K, K + 1)
                  if abs(i) + abs(j) + abs(k) <= K])
    n, M = len(rx), len(I)
    far = I * ROOM + np.where(I % 2 == 0, rx[:, None, :], ROOM - rx[:, None, :])
    ray = far - tx
    ax, plane, there = np.zeros((M, K), int), np.zeros((M, K), int), np.zeros((M, K), bool)
    for p, idx in enumerate(I):
        walls = [(a, q if idx[a] > 0 else 1 - q) for a in range(3) for q in range(1, abs(idx[a]) + 1)]
        for s, (a, q) in enumerate(walls):
            ax[p, s], plane[p, s], there[p, s] = a, q, True
    m = np.arange(M)[:, None]
    with np.errstate(divide="ignore", invalid="ignore"):
        t = (plane * ROOM[ax] - tx[ax]) / ray[:, m, ax]
    t = np.where(there, t, np.inf)
    o = np.argsort(t, axis=2)
    t = np.take_along_axis(t, o, 2)
    ax, plane, there = (np.take_along_axis(np.broadcast_to(x, (n, M, K)), o, 2) for x in (ax, plane, there))
    u = tx + np.where(there, t, 0.0)[..., None] * ray[:, :, None, :]
    cell = np.floor(u / ROOM)
    pts = np.where(cell % 2 == 0, u - cell * ROOM, (cell + 1) * ROOM - u)
    hit = np.where(plane % 2 == 1, ROOM[ax], 0.0)
    pts = np.where(np.arange(3) == ax[..., None], hit[..., None], pts)
    seq = np.full((n * M, 8), -1)
    seq[:, :K] = np.where(there, 2 * ax + plane % 2, -1).reshape(n * M, K)
    P = np.zeros((n * M, 8, 3))
    P[:, :K] = np.where(there[..., None], pts, 0.0).reshape(n * M, K, 3)
    r, nb = np.repeat(np.arange(n), M), np.tile(np.abs(I).sum(1), n)
    order = np.lexsort(tuple(seq[:, k] for k in range(7, -1, -1)) + (nb, r))
    return dict(rx=r[order], nb=nb[order], seq=seq[order], pts=P[order],
                L=np.linalg.norm(ray, axis=2).reshape(-1)[order], M=M)


def _room_case(case, seed):
    """Ends, materials, frequencies and arrays of a synth, elements or targets case (host)."""
    rng = np.random.default_rng([seed, 11])
    kind, F = case["kind"], case["F"]
    fc = 100e9
    tx = np.array([0.5, 4.0, 2.0]) + rng.uniform(-0.3, 0.3, 3)
    rx0 = np.array([8.5, 3.0, 1.2]) + rng.uniform(-0.5, 0.5, 3)
    c = dict(mats=_materials(rng, 6), tx=tx, rx=rx0[None, :], freqs=_grid(fc, F))
    if kind == "targets":
        c["rx"] = rng.uniform(0.2, 1.0, (case["n_rx"], 3)) * (ROOM - 0.3)
        c["freqs"] = np.linspace(0.9 * fc, 1.1 * fc, F)
    elif kind == "elements":
        c["rx"] = _ula(rx0, case["Nr"], 0.08)
    c["gamma"] = (0.5 + 0.1 * (c["freqs"] - fc) / 5e9).astype(np.float32)
    if kind != "targets":
        c["tx_elem"], c["rx_elem"] = _upa(tx, case["Nt"], C0 / fc / 2), _ula(rx0, case["Nr"], C0 / fc / 2)
    return c


# ---------------------------------------------------------------- prepare
def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def _prepare_link(case, seed):
    rng = np.random.default_rng([seed, 7])
    s = dict(kind="link", K=case["K"], N=case["N"], sah=case["sah"], pol=sbr.POL_V if case["pol"] == "V" else sbr.POL_H)
    if case["scene"] == "street":
        groups = [_face(2, 0.0, np.array([-20.0, 80.0]), np.array([-30.0, 70.0]))] + _box((30, 35, 0), (50, 45, 15), 1)
        s["tx"], rx, fc, gamma = np.array([0, 0, 10.0]) + rng.uniform(-2, 2, 3), np.array([[60.0, 25, 1.5]]) + rng.uniform(-1, 1, (1, 3)), 28e9, 0.1
        mats = np.tile([5.31, 0.48, 0.0], (len(groups), 1))
    elif case["scene"] == "room":
        groups = _furnished(rng)
        s["tx"], rx, fc, gamma = np.array([0.5, 4.0, 2.0]) + rng.uniform(-0.2, 0.2, 3), np.array([[8.5, 3.0, 1.2]]) + rng.uniform(-0.2, 0.2, (1, 3)), 100e9, 0.5
        mats = _materials(rng, len(groups))
    else:
        ground = 40 if case["tri"] > 20000 else 8
        groups = _city(rng, 8, 5, max(1, round(math.sqrt((case["tri"] - 2 * ground * ground) / 400))) if case["tri"] > 2 * ground * ground else 1, ground)
        side = math.ceil(math.sqrt(case["n_rx"]))
        g = (np.arange(side) - (side - 1) / 2) * 2.0
        c = np.array([240.0, 120.0]) + rng.uniform(-3, 3, 2)
        rx = np.array([(c[0] + x, c[1] + y, 1.5) for x in g for y in g])[:case["n_rx"]]
        s["tx"], fc, gamma = np.array([c[0], c[1], rng.uniform(20, 30)]), 300e9, 5.0
        mats = _materials(rng, len(groups))
    f = _grid(fc, case["F"]) if case["F"] > 1 else np.array([fc])
    s["tri"], s["sid"] = _mesh(groups)
    s.update(S=len(groups), fc=fc, f_mid=case["F"] // 2, tx=[float(x) for x in s["tx"]], rx=_dev(rx, torch.float64),
             mats=_dev(mats, torch.float64), freqs=_dev(f, torch.float64), gamma=_dev(gamma * f / fc, torch.float32),
             siso=case["scene"] == "street", bins=2048 if case["scene"] == "urban" else 512)
    s["tx_elem"], s["rx_elem"] = _dev([s["tx"]], torch.float64), s["rx"][:1].contiguous()
    # result buffers that a program keeps from one scene to the next; rows after the last path stay zero
    rows = s["rows"] = 256 + 64 * case["n_rx"]
    shape = dict(rx=((), torch.int32), nb=((), torch.int32), seq=((8,), torch.int32), face=((8,), torch.int32), pts=((8, 3), torch.float64),
                 L=((), torch.float64), aod=((2,), torch.float64), aoa=((2,), torch.float64), ray=((), torch.int32), dist=((), torch.float32))
    s["out"] = {k: torch.zeros((rows,) + sh, dtype=dt, device="cuda") for k, (sh, dt) in shape.items()}
    s["g"] = torch.zeros(rows, case["F"], dtype=torch.complex64, device="cuda")
    return s


def _prepare_room(case, seed):
    c = _room_case(case, seed)
    tri, sid = _mesh(_box((0, 0, 0), tuple(ROOM), 2))
    p = room_paths(c["tx"], c["rx"], case["K"])
    keys = np.full((len(p["nb"]), 10), -1, np.int64)
    keys[:, 0], keys[:, 1], keys[:, 2:] = p["rx"], p["nb"], p["seq"]
    vals = (p["L"].astype(np.float32).view(np.int32).astype(np.int64) << 32) | np.arange(len(p["nb"]))
    rx = _dev(c["rx"], torch.float64)
    bvh = sbr.build_bvh(tri, sid, 6)
    pl = sbr.paths(sbr.trace_merge([float(x) for x in c["tx"]], rx, 100, case["K"], _dev(keys, torch.int32), _dev(vals, torch.int64)), bvh)
    if pl.n != len(p["nb"]):
        raise RuntimeError("%d of %d paths of the room" % (pl.n, len(p["nb"])))
    s = dict(kind=case["kind"], bvh=bvh, pl=pl, mats=_dev(c["mats"], torch.float64), freqs=_dev(c["freqs"], torch.float64),
             gamma=_dev(c["gamma"], torch.float32), pol=sbr.POL_V if case["pol"] == "V" else sbr.POL_H, F=case["F"])
    if case["kind"] != "targets":
        s["g"] = sbr.path_gains(pl, s["mats"], s["freqs"], s["gamma"], None, s["pol"])
        s["tx_elem"], s["rx_elem"], s["precision"] = _dev(c["tx_elem"], torch.float64), _dev(c["rx_elem"], torch.float64), PRECISION[case["precision"]]
    return s


def _capacity_inputs(case, seed):
    """H(f) of 40 plane-wave paths with delays, at an indoor link's level, plus what is too weak to be resolved."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    F, Nr, Nt = case["F"], case["Nr"], case["Nt"]

    def uniform(*shape):
        return torch.rand(shape, device="cuda", generator=g)

    def wave(n):
        return torch.polar(torch.ones(n, 40, device="cuda"), math.pi * torch.arange(n, device="cuda")[:, None] * (2 * uniform(1, 40) - 1))

    amp = 1e-5 * 10 ** (-1.5 * uniform(40))
    w = torch.polar(amp.expand(F, 40).contiguous(), 2 * math.pi * (uniform(40) + torch.linspace(0, 40, F, device="cuda")[:, None] * uniform(40)))
    H = torch.einsum("fn,rn,tn->frt", w, wave(Nr), wave(Nt))
    noise = torch.randn(F, Nr, Nt, 2, device="cuda", generator=g)
    return (H + 1e-8 * torch.view_as_complex(noise)).contiguous(), [5.0 * k for k in range(case["n_snr"])]


def _prepare_capacity(case, seed):
    H, snr = _capacity_inputs(case, seed)
    return dict(kind="capacity", H=H, snr=snr)


X_LO, X_HI = (-20.0, -20.0, 0.0, 280e9), (500.0, 320.0, 10.0, 320e9)
SHIFT, SCALE = [120.0, 20.0] + [-20.0] * N_TAPS + [0.0, 0.0], [20.0] * (2 + N_TAPS) + [1.0, 20.0]
LOSS_W, FEAT, LR = [1.0, 0.5] + [0.25] * N_TAPS + [1.0, 0.5], 2.5, 5e-4


def _network(case, seed):
    """Weights (flat, per layer W then b), queries and targets of a surrogate network."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    dims = [128] + [case["width"]] * case["depth"] + [128]
    w = torch.cat([t for i, o in zip(dims[:-1], dims[1:])
                   for t in ((2 * torch.rand(o * i, device="cuda", generator=g) - 1) * math.sqrt(6 / i),
                             0.05 * torch.randn(o, device="cuda", generator=g))])
    B = case["B"]
    u = torch.rand(B, 4, device="cuda", generator=g)
    lo, hi = torch.tensor(X_LO, device="cuda"), torch.tensor(X_HI, device="cuda")
    y = None
    if case["kind"] == "train":   # smooth in position, some receivers without coverage
        a = torch.randn(4, N_OUT, device="cuda", generator=g)
        y = torch.tensor(SHIFT, device="cuda") + torch.tensor(SCALE, device="cuda") * torch.sin(3 * u @ a)
        covered = torch.sin(9 * u[:, 0]) + torch.sin(7 * u[:, 1]) > -0.3
        y[~covered, :18] = float("nan")
        y[:, 18] = covered.float()
        y[:, 19] = float("nan")
    return dims, w, lo + u * (hi - lo), y


def _prepare_net(case, seed):
    dims, w, x, y = _network(case, seed)
    m = sbr.MLP(N_OUT, X_LO, X_HI, width=case["width"], depth=case["depth"], max_batch=case["B"], seed=1, lr=LR,
                err_channel=19, err_of=0, loss_w=LOSS_W, y_shift=SHIFT, y_scale=SCALE, feat_log2_max=FEAT)
    m.params(1, w)
    return dict(kind=case["kind"], m=m, x=x.contiguous(), y=y)


def _prepare_batch(case, seed):
    rng = np.random.default_rng([seed, 13])
    scs = []
    for _ in range(case["scenes"]):
        nx, ny = int(rng.integers(3, 9)), int(rng.integers(2, 6))
        groups = _city(rng, nx, ny, max(1, round(math.sqrt(case["tri"] * math.exp(rng.uniform(-1, 0.3)) / (10 * nx * ny)))), 8)
        tri, sid = _mesh(groups)
        scs.append((sbr.build_bvh(tri, sid, len(groups), sah_top=True), _dev(_materials(rng, len(groups)), torch.float64), nx, ny))
    jobs = []
    ns = np.geomspace(case["n_min"], case["n_max"], case["jobs"])   # ray counts spread evenly over the range
    for k in range(case["jobs"]):
        i = int(rng.integers(0, len(scs)))
        nx, ny = scs[i][2:]
        fc = float(rng.choice([28e9, 60e9, 100e9, 140e9, 300e9]))
        f = _grid(fc, max(64, case["f_max"] >> (k % 5)))
        tx = np.array([60.0 * rng.integers(1, nx) + rng.uniform(-5, 5), 60.0 * rng.integers(1, ny) + rng.uniform(-5, 5), rng.uniform(5, 30)])
        rx = np.array([60.0 * rng.integers(0, nx + 1) + rng.uniform(-8, 8), rng.uniform(-10.0, 60.0 * ny + 10.0), 1.5])
        jobs.append(dict(scene=i, N=int(round(ns[k])), K=2 + k % 7, tx=tx, rx=rx, pol="VH"[k % 2], freqs=_dev(f, torch.float64),
                         gamma=_dev(5.0 * f / 300e9, torch.float32), tx_elem=_dev(_upa(tx, 1 << (5 * k % 7), C0 / fc / 2), torch.float64),
                         rx_elem=_dev(_ula(rx, 1 << (3 * k % 7), C0 / fc / 2), torch.float64)))
    b = sbr.batch_create([s[:2] for s in scs], jobs, config=dict(wave_rays=1 << 28, path_cap=256))
    return dict(kind="batch", b=b, H=[j["H"] for j in jobs])


_PREPARE = dict(link=_prepare_link, synth=_prepare_room, elements=_prepare_room, targets=_prepare_room,
                capacity=_prepare_capacity, train=_prepare_net, predict=_prepare_net, batch=_prepare_batch)


# ---------------------------------------------------------------- run
def run(s):
    kind = s["kind"]
    if kind == "link":
        bvh = sbr.build_bvh(s["tri"], s["sid"], s["S"], sah_top=s["sah"])
        pl = sbr.paths(sbr.trace(bvh, s["tx"], s["rx"], s["N"], s["K"]), bvh)
        if pl.n > s["rows"]:
            raise RuntimeError("%d paths in buffers of %d" % (pl.n, s["rows"]))
        g = sbr.path_gains(pl, s["mats"], s["freqs"], s["gamma"], None, s["pol"], out=s["g"])
        out = dict(paths=pl.export(out=s["out"]), g=g)
        out["pdp"], out["stats"] = sbr.pdp_angles(pl, g, s["f_mid"], s["fc"], 1e-9, s["bins"])
        if s["siso"]:
            out["H"] = sbr.synthesize_H(pl, g, s["freqs"], s["tx_elem"], s["rx_elem"])
        return out
    if kind == "synth":
        return sbr.synthesize_H(s["pl"], s["g"], s["freqs"], s["tx_elem"], s["rx_elem"], 0, s["precision"])
    if kind == "elements":
        return sbr.synthesize_H_elements(s["pl"], s["g"], s["freqs"], s["tx_elem"], s["precision"])
    if kind == "capacity":
        return sbr.capacity(s["H"], s["snr"])
    if kind == "targets":
        g = sbr.path_gains(s["pl"], s["mats"], s["freqs"], s["gamma"], None, s["pol"])
        return g, sbr.surrogate_targets(s["pl"], g, s["F"], N_TAPS, TAP_S, FLOOR_DB)
    if kind == "train":
        loss = torch.zeros(1, device="cuda")
        s["m"].train_step(s["x"], s["y"], loss)
        return dict(loss=loss, grad=s["m"].params(2), weights=s["m"].params(0))
    if kind == "predict":
        return s["m"].predict(s["x"])
    s["b"].run()
    return s["H"]


# ---------------------------------------------------------------- work
def work(case):
    """Inputs once, outputs once; operations as counted in the comments."""
    kind = case["kind"]
    if kind == "link":
        rays, T = 10 * case["N"] ** 2 + 2, case["tri"]
        seg = rays * (1 + 0.25 * case["K"])             # outdoors most rays escape at once; each segment goes down the tree once
        paths = 8 * case["n_rx"]
        return dict(bytes=40 * T + 24 * case["n_rx"] + paths * (240 + 8 * case["F"]) + 8192 * case["n_rx"],
                    flops=seg * (2 * 24 * math.log2(T) + 60) + paths * case["F"] * 200 * case["K"])
    if kind in ("synth", "elements"):
        M = _room_count(case["K"])
        F, Nr, Nt = case["F"], case["Nr"], case["Nt"]
        P = M * (Nr if kind == "elements" else 1)
        phasors = P * Nt * F if kind == "elements" else M * (Nr + Nt) * F
        return dict(bytes=8 * F * Nr * Nt + 8 * P * F + 200 * P + 24 * (Nt + Nr), flops=8.0 * F * Nr * Nt * M + 20.0 * phasors)
    if kind == "capacity":
        F, a, b = case["F"], min(case["Nr"], case["Nt"]), max(case["Nr"], case["Nt"])
        return dict(bytes=8 * F * a * b + 8 * case["n_snr"], flops=F * (4.0 * a * a * b + case["n_snr"] * (4 / 3) * a ** 3))
    if kind == "targets":
        n, F, M = case["n_rx"], case["F"], _room_count(case["K"])
        return dict(bytes=n * M * (8 * F + 360) + 4 * n * F * (2 + N_TAPS), flops=n * M * F * (200.0 * case["K"] + 40))
    if kind in ("train", "predict"):
        d = [128] + [case["width"]] * case["depth"] + [128]
        w = sum(i * o for i, o in zip(d[:-1], d[1:]))
        B = case["B"]
        if kind == "predict":
            return dict(bytes=2 * w + B * (16 + 4 * N_OUT), flops=2.0 * w * B + 64 * 20 * B)
        return dict(bytes=w * (4 * 7 + 2 * 4) + B * (16 + 4 * N_OUT), flops=3 * 2.0 * w * B + 64 * 20 * B)
    ns = np.geomspace(case["n_min"], case["n_max"], case["jobs"])
    rays = float(np.sum(10 * ns ** 2 + 2))
    h = sum(max(64, case["f_max"] >> (k % 5)) << (5 * k % 7 + 3 * k % 7) for k in range(case["jobs"]))   # elements of all H
    return dict(bytes=8 * h + 40 * case["tri"] * case["scenes"], flops=2.0 * rays * (2 * 24 * math.log2(case["tri"]) + 60) + 8 * 4 * h)


def _room_count(K):
    return 1 + sum(4 * k * k + 2 for k in range(1, K + 1))


# ---------------------------------------------------------------- exact
def exact(case, seed):
    """None for link and batch: which rays reach a receiver has no closed form in their scenes."""
    f = dict(synth=_exact_synth, elements=_exact_elements, targets=_exact_targets, capacity=_exact_capacity,
             train=_exact_train, predict=_exact_predict).get(case["kind"])
    return f(case, seed) if f else None


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _polar_vector(d, pol):
    r = torch.hypot(d[:, 0], d[:, 1])
    cp, sp = d[:, 0] / r, d[:, 1] / r
    return torch.stack([d[:, 2] * cp, d[:, 2] * sp, -r] if pol == "V" else [-sp, cp, torch.zeros_like(r)], 1)


def _exact_gains(case, c, p):
    """Complex gains [P, F]: Fresnel coefficients and roughness of every reflection on the vector field, spreading, absorption."""
    f, nb = _d(c["freqs"]), torch.as_tensor(p["nb"], device="cuda")
    pts, tx, rx, L = _d(p["pts"]), _d(c["tx"]), _d(c["rx"])[torch.as_tensor(p["rx"], device="cuda")], _d(p["L"])
    K = int(case["K"])

    def corner(k):   # point k of every path: the transmitter, the reflections, then the receiver
        inner = pts[:, k - 1] if 1 <= k <= K else tx.expand(len(nb), 3)
        return tx.expand(len(nb), 3) if k == 0 else torch.where((k > nb)[:, None], rx, inner)

    d = _unit(corner(1) - corner(0))
    E = _polar_vector(d, case["pol"])[:, None, :].to(torch.complex128).expand(-1, len(f), -1)
    for k in range(1, K + 1):
        on = torch.nonzero(nb >= k)[:, 0]
        wall = torch.as_tensor(p["seq"][:, k - 1], device="cuda")[on]
        n = torch.nn.functional.one_hot(wall // 2, 3).double()
        mat = _d(c["mats"])[wall]
        din, dout = d[on], _unit(corner(k + 1)[on] - corner(k)[on])
        s = _unit(torch.linalg.cross(din, n))
        pin, pout = torch.linalg.cross(s, din), torch.linalg.cross(s, dout)
        cos = (din * n).sum(1).abs()[:, None]
        eta = torch.complex(mat[:, 0:1].expand(-1, len(f)), -mat[:, 1:2] / (2 * math.pi * f * EPS0))
        root = torch.sqrt(eta - (1 - cos * cos))
        te, tm = (cos - root) / (cos + root), (eta * cos - root) / (eta * cos + root)
        rho = torch.exp(-0.5 * (4 * math.pi * f / C0 * mat[:, 2:3] * cos) ** 2)
        e = E[on]
        e = rho[..., None] * ((te * (e * s[:, None]).sum(-1))[..., None] * s[:, None] + (tm * (e * pin[:, None]).sum(-1))[..., None] * pout[:, None])
        E = E.index_copy(0, on, e)
        d = d.index_copy(0, on, dout)
    g = (E * _polar_vector(d, case["pol"])[:, None, :]).sum(-1)
    return g * C0 / (4 * math.pi * f * L[:, None]) * 10 ** (-_d(c["gamma"].astype(np.float64)) * L[:, None] / 20000)


def _rotate(f, length):
    cyc = f * (length / C0)
    return torch.polar(torch.ones_like(cyc), -2 * math.pi * (cyc - torch.floor(cyc)))


def _exact_synth(case, seed):
    c = _room_case(case, seed)
    p = room_paths(c["tx"], c["rx"], case["K"])
    g, f, L = _exact_gains(case, c, p), _d(c["freqs"]), _d(p["L"])
    T, R, t0, r0 = _d(c["tx_elem"]), _d(c["rx_elem"]), _d(c["tx"]), _d(c["rx"][0])
    first, last = _d(p["pts"][1:, 0]), _d(p["pts"][np.arange(1, len(L)), p["nb"][1:] - 1])
    dt = (T - first[:, None]).norm(dim=-1) - (t0 - first).norm(dim=-1)[:, None]
    dr = (R - last[:, None]).norm(dim=-1) - (r0 - last).norm(dim=-1)[:, None]
    los = (T - R[:, None]).norm(dim=-1)
    H = torch.empty(case["F"], case["Nr"], case["Nt"], dtype=torch.complex128, device="cuda")
    for k in range(0, case["F"], 64):
        ff = f[k:k + 64, None, None]
        w = g[1:, k:k + 64].T * _rotate(ff[..., 0], L[1:])
        H[k:k + 64] = torch.matmul(_rotate(ff, dr.T) * w[:, None, :], _rotate(ff, dt)) + g[0, k:k + 64, None, None] * _rotate(ff, los)
    return H


def _exact_elements(case, seed):
    c = _room_case(case, seed)
    p = room_paths(c["tx"], c["rx"], case["K"])
    M, Nr, Nt = p["M"], case["Nr"], case["Nt"]
    g, f, L = _exact_gains(case, c, p).reshape(Nr, M, -1), _d(c["freqs"]), _d(p["L"]).reshape(Nr, M, 1)
    T, t0 = _d(c["tx_elem"]), _d(c["tx"])
    first = _d(p["pts"][:, 0]).reshape(Nr, M, 1, 3)
    length = L + (T - first).norm(dim=-1) - (t0 - first).norm(dim=-1)
    length[:, 0] = (T - _d(c["rx"])[:, None]).norm(dim=-1)   # the path without reflections comes first
    H = torch.empty(case["F"], Nr, Nt, dtype=torch.complex128, device="cuda")
    for k in range(0, case["F"], 8):
        ff = f[k:k + 8, None, None, None]
        H[k:k + 8] = (g[..., k:k + 8].permute(2, 0, 1)[..., None] * _rotate(ff, length)).sum(2)
    return H


def _exact_targets(case, seed):
    c = _room_case(case, seed)
    p = room_paths(c["tx"], c["rx"], case["K"])
    n, F, M = case["n_rx"], case["F"], p["M"]
    g, L = _exact_gains(case, c, p), _d(p["L"]).reshape(n, M)
    pw = (g.real ** 2 + g.imag ** 2).reshape(n, M, F)
    t = (L - L.min(1, keepdim=True).values) / C0
    total = pw.sum(1)
    mean = (pw * t[..., None]).sum(1) / total
    spread = torch.sqrt(torch.clamp((pw * (t * t)[..., None]).sum(1) / total - mean * mean, min=0.0))
    b = torch.floor(t / TAP_S).long()
    w = torch.where((b < N_TAPS)[..., None], pw, torch.zeros_like(pw))
    taps = torch.zeros(n, N_TAPS, F, dtype=torch.float64, device="cuda").scatter_add(1, b.clamp(max=N_TAPS - 1)[..., None].expand(n, M, F), w)
    db = torch.clamp(10 * torch.log10(taps / total[:, None]), min=FLOOR_DB).transpose(1, 2)
    return g, torch.cat([-10 * torch.log10(total)[..., None], spread[..., None], db], 2)


def _exact_capacity(case, seed):
    H, snr = _capacity_inputs(case, seed)
    H = H.to(torch.complex128)
    F, Nr, Nt = H.shape
    W = H @ H.mH if Nt >= Nr else H.mH @ H
    W = (W * (Nr * Nt / (H.abs() ** 2).sum((1, 2)).mean())).cpu()
    eye = torch.eye(W.shape[1], dtype=torch.complex128)
    logdet = [2 * torch.log2(torch.linalg.cholesky(eye + 10 ** (x / 10) / Nt * W).diagonal(dim1=1, dim2=2).real).sum(1) for x in snr]
    return torch.stack([x.mean() for x in logdet])


def _forward(dims, w, x):
    u = (x.double() - _d(X_LO)) / (_d(X_HI) - _d(X_LO))
    a = math.pi * 2.0 ** (FEAT * torch.arange(16, device="cuda", dtype=torch.float64) / 15) * u[:, :, None]
    h, at = torch.stack([torch.sin(a), torch.cos(a)], 3).reshape(len(x), 128), 0
    for k, (i, o) in enumerate(zip(dims[:-1], dims[1:])):
        h = h @ w[at:at + i * o].reshape(o, i).T + w[at + i * o:at + i * o + o]
        at += i * o + o
        h = torch.relu(h) if k + 2 < len(dims) else h
    return h[:, :N_OUT]


def _exact_predict(case, seed):
    dims, w, x, _ = _network(case, seed)
    w = w.double()
    return torch.cat([_forward(dims, w, x[k:k + 65536]) * _d(SCALE) + _d(SHIFT) for k in range(0, len(x), 65536)])


def _exact_train(case, seed):
    dims, w, x, y = _network(case, seed)
    w = w.double().requires_grad_(True)
    out, t = _forward(dims, w, x), (y.double() - _d(SHIFT)) / _d(SCALE)
    head = (out[:, 0] - t[:, 0]).abs().detach()
    t = torch.cat([t[:, :19], head[:, None]], 1)
    on = torch.isfinite(t)
    loss = ((out - torch.where(on, t, torch.zeros_like(t))) ** 2 * _d(LOSS_W))[on].sum() / len(x)
    grad, = torch.autograd.grad(loss, w)
    return dict(loss=loss.detach().reshape(1), grad=grad, weights=(w - LR * grad / (grad.abs() + 1e-8)).detach())

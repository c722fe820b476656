"""Timed cases of the library: what a user of the hybrid Monte Carlo method has it do.

Each case goes through the public binding (``paper_1007_3509_gb300.hmcpotts``) the way the
drivers in ``hybrid.py`` and ``texture.py`` and the workloads of ``bench.py`` call it.  A pass
starts from the same state every time (the initial lattice is loaded with ``hp_set_spins``, the
plasticity state with ``hp_cp_reset``, the network from its initial weights), so that one pass
costs what the next one does: a lattice swept on and on coarsens until nothing is left to sweep.
Sizes are those of the workload presets in ``synth.py``, of the tests and of the bench, or lie
between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1007_3509_gb300 import hmcpotts as hm
from paper_1007_3509_gb300 import synth
from paper_1007_3509_gb300.hybrid import cp_params_table1

NI = (synth.NI_BJ["C11"], synth.NI_BJ["C12"], synth.NI_BJ["C44"])
GROUP = 20                      # training rows per orientation (load increments)
LR, LR_FLOOR = 3e-3, 0.02       # the surrogate's training schedule
EPS_P = 1e-4                  # plastic strain scale handed to the elastic solve


# ------------------------------------------------------------------------------------------------
# Cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest run: one 128^2 lattice, 100 MCS in one call; launches and latency count
        dict(name="sweep-2d-128", kind="sweep", dim=2, nbr=4, x=128, y=128, z=1, grains=64, kT=0.5, mcs=100,
             field="grain"),
        # the 2D Moore workload: 10^4 grains, closed-form grain energies
        dict(name="sweep-2d-4096", kind="sweep", dim=2, nbr=8, x=4096, y=4096, z=1, grains=10_000, kT=0.6, mcs=20,
             field="grain"),
        # a 3D lattice whose edges fit no tile (250 is no multiple of 4), material points carried
        dict(name="sweep-3d-ragged", kind="sweep", dim=3, nbr=26, x=250, y=198, z=130, grains=6_000, kT=0.7, mcs=10,
             field="point"),
        # the plasticity-driven hybrid: refresh the field at every material point, sweep, measure
        dict(name="hybrid-3d-512", kind="hybrid", x=512, y=512, z=512, grains=200_000, kT=0.7, mcs=10),
        # the surrogate-driven hybrid at full size: network once per grain, then sweep
        dict(name="surrogate-3d-1024", kind="surrogate", x=1024, y=1024, z=1024, grains=1_000_000, kT=0.7, mcs=3),
        # independent 3D replicas of uneven size, temperature and load in one launch, tile autotuned
        dict(name="ensemble-3d-24", kind="ensemble3d", replicas=24, edge_max=256, mcs=5),
        # the 2D texture experiment (Gaussian grain energies): one time slice, then measure all members
        dict(name="texture-2d-32x500", kind="ensemble2d", replicas=32, x=500, y=500, grains=5000, kT=1.0, mcs=100),
        # Read-Shockley pair energies and mobilities on a Moore lattice
        dict(name="aniso-2d-1024", kind="aniso", x=1024, y=1024, grains=625, kT=0.6, mcs=20),
        # Monte Carlo plasticity on its own: a load path of 20 increments, every output asked for
        dict(name="plasticity-1e6x20", kind="plasticity", points=1_000_000, grains=4096, incr=20),
        # training of the field network: Adam steps on minibatches of whole orientations (a short
        # call: after some fifty steps the rounding of two runs of the same training shows in the moments)
        dict(name="train-19440x32", kind="train", batch=19440, steps=32),
        # periodic elastic equilibrium of the polycrystal under one load increment
        dict(name="elastic-256", kind="elastic", x=256, y=256, z=256, grains=15_625, iters=8),
        # the initial polycrystal
        dict(name="voronoi-3d-256", kind="voronoi", dim=3, x=256, y=256, z=256, grains=16_000),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    return max(2, 2 * int(round(_log(rng, lo, hi) / 2)))


def draw(rng):
    kind = rng.choice(["sweep2d", "sweep2d", "sweep3d", "sweep3d", "hybrid", "surrogate", "ensemble3d", "ensemble2d",
                       "aniso", "plasticity", "train", "elastic", "voronoi"])
    if kind == "sweep2d":
        x, y = _even(rng, 64, 4096), _even(rng, 64, 4096)
        return dict(kind="sweep", dim=2, nbr=rng.choice([4, 8]), x=x, y=y, z=1, grains=int(max(8, x * y / _log(rng, 200, 3000))),
                    kT=round(rng.uniform(0.4, 1.0), 3), mcs=rng.randint(5, 100 if x * y < 1 << 20 else 20),
                    field=rng.choice(["grain", "grain", "point"]))
    if kind == "sweep3d":
        x, y, z = _even(rng, 40, 512), _even(rng, 40, 512), _even(rng, 8, 256)
        return dict(kind="sweep", dim=3, nbr=rng.choice([26, 26, 26, 6]), x=x, y=y, z=z,
                    grains=int(max(8, x * y * z / _log(rng, 400, 3000))), kT=round(rng.uniform(0.5, 0.9), 3),
                    mcs=rng.randint(2, 8), field=rng.choice(["grain", "point"]))
    if kind in ("hybrid", "surrogate"):
        x, y, z = _even(rng, 64, 512), _even(rng, 64, 512), _even(rng, 32, 384)
        return dict(kind=kind, x=x, y=y, z=z, grains=int(max(8, x * y * z / _log(rng, 500, 3000))),
                    kT=round(rng.uniform(0.5, 0.9), 3), mcs=rng.randint(2, 10))
    if kind == "ensemble3d":
        return dict(kind=kind, replicas=rng.randint(3, 24), edge_max=rng.choice([96, 128, 192, 256]), mcs=rng.randint(1, 5))
    if kind == "ensemble2d":
        x = _even(rng, 100, 600)
        return dict(kind=kind, replicas=rng.randint(4, 32), x=x, y=x, grains=max(20, x * x // 50),
                    kT=round(rng.uniform(0.6, 1.2), 3), mcs=rng.randint(20, 100))
    if kind == "aniso":
        x, y = _even(rng, 128, 1500), _even(rng, 128, 1500)
        return dict(kind=kind, x=x, y=y, grains=int(max(8, x * y / _log(rng, 400, 3000))),
                    kT=round(rng.uniform(0.4, 0.8), 3), mcs=rng.randint(5, 20))
    if kind == "plasticity":
        return dict(kind=kind, points=int(_log(rng, 3000, 2e6)), grains=rng.randint(16, 8192), incr=rng.randint(1, 20))
    if kind == "train":
        return dict(kind=kind, batch=GROUP * int(_log(rng, 50, 1500)), steps=rng.randint(8, 32))
    if kind == "elastic":
        x, y, z = (1 << rng.randint(4, 8) for _ in range(3))
        return dict(kind=kind, x=x, y=y, z=z, grains=int(max(4, x * y * z / 1000)), iters=rng.randint(4, 8))
    if rng.random() < 0.3:
        x, y, z, dim = _even(rng, 128, 4096), _even(rng, 128, 4096), 1, 2
    else:
        x, y, z, dim = _even(rng, 48, 320), _even(rng, 48, 320), _even(rng, 32, 256), 3
    return dict(kind="voronoi", dim=dim, x=x, y=y, z=z, grains=int(max(8, x * y * z / _log(rng, 300, 4000))))


def _sites(c):
    return c["x"] * c["y"] * c.get("z", 1)


def _members3d(c):
    """Edges, temperatures, loads and grain counts of the replicas (the same for every seed)."""
    rng = np.random.default_rng(1000 + c["replicas"])
    edges = [e for e in (64, 96, 128, 192, 256) if e <= c["edge_max"]]
    out = []
    for _ in range(c["replicas"]):
        e = int(rng.choice(edges))
        out.append(dict(edge=e, kT=float(rng.uniform(0.5, 0.9)), sigma=float(rng.uniform(50.0, 200.0)),
                        G=int(min(rng.integers(500, 20_001), e ** 3 // 200))))
    return out


# ------------------------------------------------------------------------------------------------
# Inputs and handles
# ------------------------------------------------------------------------------------------------
def _i32(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _f32(n):
    return torch.empty(n, dtype=torch.float32, device="cuda")


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _quats(n, seed):
    q = torch.randn(n, 4, generator=_gen(seed), device="cuda", dtype=torch.float32)
    return (q / q.norm(dim=1, keepdim=True)).contiguous()


def _lattice(dim, L, nbr, G, seed, mode, mp, kT, orient):
    """A bound handle holding a seeded polycrystal, and the lattice's initial ids."""
    n = int(np.prod(L))
    lat = hm.Lattice(dim, L, nbr, 256, seed, G, mode)
    q = _i32(n)
    m = _i32(n) if mp else None
    lat.hp_bind(q, m)
    lat.hp_init_voronoi(hm.ORIENT_ANGLE if orient.dim() == 1 else hm.ORIENT_SO3, orient)
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    return lat, q, m, q.clone()


def _grain_energies(quat, sigma=100.0):
    b = _i32(quat.shape[0])
    hm.hp_grain_field(quat, *NI, sigma, 0.05, 1.0, b)
    return b


def _cp_state(n):
    return dict(eps=_f32(6 * n), gam=_f32(n), g=_f32(n), b=_i32(n))


def _net(seed):
    w = np.concatenate([p.ravel() for p in synth.mlp_init(int(seed) & 0x7FFFFFFF)]).astype(np.float32)
    return torch.from_numpy(w).cuda()


def _train_data(c, seed):
    """Orientation-major rows as hp_sur_generate lays them out: four invariants of the loading
    axis, a load path of GROUP increments (stress, slip), smooth targets of order one."""
    orients = (4 * c["batch"] + GROUP - 1) // GROUP
    d = torch.randn(orients, 3, generator=_gen(seed), device="cuda", dtype=torch.float64)
    d = (d / d.norm(dim=1, keepdim=True)).abs().sort(dim=1, descending=True).values
    inv = (d[:, 0] * d[:, 1]) ** 2 + (d[:, 1] * d[:, 2]) ** 2 + (d[:, 2] * d[:, 0]) ** 2
    t = (torch.arange(1, GROUP + 1, device="cuda", dtype=torch.float64) / GROUP)
    s = 0.5 * torch.tanh(3.0 * t)
    load = torch.stack([s, -0.5 * s, -0.5 * s, 0.01 * t, -0.02 * t, 0.01 * t * t, 3.0 * t], dim=1)
    X = torch.cat([d, inv[:, None]], dim=1)[:, None, :].expand(orients, GROUP, 4)
    X = torch.cat([X, load[None].expand(orients, GROUP, 7)], dim=2).reshape(-1, 11)
    f = X[:, 3] * (1.0 + X[:, 4]) + 0.3 * X[:, 0]
    h = 0.2 + 0.4 * X[:, 10] * (1.0 + 0.5 * X[:, 3])
    return X.to(torch.float32).contiguous(), torch.stack([f, h], dim=1).to(torch.float32).contiguous()


def _plastic_inputs(c, seed):
    P, G = c["points"], c["grains"]
    grain = torch.randint(0, G, (P,), generator=_gen(seed), device="cuda", dtype=torch.int32)
    return grain, _quats(G, seed + 1)


def _elastic_inputs(c, seed):
    """Blocky polycrystal (about ten voxels per grain edge), random plastic strain, a Taylor-type load."""
    n, G = (c["x"], c["y"], c["z"]), c["grains"]
    coarse = [max(1, v // 10) for v in n]
    cg = torch.randint(0, G, tuple(reversed(coarse)), generator=_gen(seed), device="cuda", dtype=torch.int32)
    at = [torch.arange(v, device="cuda") * k // v for v, k in zip(n, coarse)]
    grain = cg[at[2][:, None, None], at[1][None, :, None], at[0][None, None, :]].reshape(-1).contiguous()
    epp = torch.randn(6, _sites(c), generator=_gen(seed + 2), device="cuda", dtype=torch.float32) * EPS_P
    return grain, _quats(G, seed + 1), epp.contiguous(), (1e-3, -5e-4, -5e-4, 0.0, 0.0, 0.0)


def prepare(case, seed):
    c, s = dict(case), {"case": dict(case)}
    kind, seed = c["kind"], int(seed)
    if kind == "sweep":
        L = (c["x"], c["y"]) if c["dim"] == 2 else (c["x"], c["y"], c["z"])
        n, G, point = _sites(c), c["grains"], c["field"] == "point"
        quat = _f32(4 * G).view(G, 4)
        lat, q, m, q0 = _lattice(c["dim"], L, c["nbr"], G, seed, hm.FIELD_POINT if point else hm.FIELD_GRAIN, point,
                                 c["kT"], quat)
        s.update(lat=lat, q=q, m=m, q0=q0, m0=None if m is None else m.clone(), keep=quat)
        if point:
            st = _cp_state(n)
            prm = cp_params_table1(1e-4, 7.0)
            hm.hp_cp_reset(prm, n, st["eps"], st["gam"], st["g"])
            hm.hp_cp_step(prm, seed, q0, quat, 0, 4, st["eps"], st["gam"], st["g"], b=st["b"])
            s["table"] = st["b"]
        elif c["nbr"] == 4:  # uniform grain energies below 0.1 J
            s["table"] = torch.randint(0, 26, (G,), generator=_gen(seed), device="cuda", dtype=torch.int32)
        else:
            s["table"] = _grain_energies(quat)
        lat.hp_set_field(s["table"])
    elif kind == "hybrid":
        L, n, G = (c["x"], c["y"], c["z"]), _sites(c), c["grains"]
        quat = _f32(4 * G).view(G, 4)
        lat, q, m, q0 = _lattice(3, L, 26, G, seed, hm.FIELD_POINT, True, c["kT"], quat)
        s.update(lat=lat, q=q, m=m, q0=q0, m0=m.clone(), quat=quat, prm=cp_params_table1(1e-4, 7.0), seed=seed,
                 **_cp_state(n))
        lat.hp_set_field(s["b"])
    elif kind == "surrogate":
        L, G = (c["x"], c["y"], c["z"]), c["grains"]
        quat = _f32(4 * G).view(G, 4)
        lat, q, _, q0 = _lattice(3, L, 26, G, seed, hm.FIELD_GRAIN, False, c["kT"], quat)
        s.update(lat=lat, q=q, m=None, q0=q0, m0=None, quat=quat, b=_i32(G), e=_f32(G), net=_net(seed),
                 load=np.array([55.0, -27.0, -28.0, 1.0, -2.0, 0.5, 2.5e-3], dtype=np.float32))
        lat.hp_set_field(s["b"])
    elif kind in ("ensemble3d", "ensemble2d"):
        members = []
        spec = _members3d(c) if kind == "ensemble3d" else [None] * c["replicas"]
        for r, p in enumerate(spec):
            if p:
                o = _f32(4 * p["G"]).view(p["G"], 4)
                lat, q, _, q0 = _lattice(3, (p["edge"],) * 3, 26, p["G"], seed + r, hm.FIELD_GRAIN, False, p["kT"], o)
                b = _grain_energies(o, p["sigma"])
            else:
                o = _f32(c["grains"])
                lat, q, _, q0 = _lattice(2, (c["x"], c["y"]), 8, c["grains"], seed + r, hm.FIELD_GRAIN, False, c["kT"], o)
                b = _i32(c["grains"])
                hm.hp_gaussian_field(c["grains"], o, 1.0, b)
            lat.hp_set_field(b)
            members.append(dict(lat=lat, q=q, m=None, q0=q0, m0=None, orient=o, b=b))
        s.update(members=members, ens=hm.Ensemble([v["lat"] for v in members]))
        if kind == "ensemble3d":
            s["ens"].hp_ensemble_autotune(1)
    elif kind == "aniso":
        G = c["grains"]
        ang = _f32(G)
        lat, q, _, q0 = _lattice(2, (c["x"], c["y"]), 8, G, seed, hm.FIELD_NONE, False, c["kT"], ang)
        units = _i32(G)
        hm.hp_angle_units(G, hm.ORIENT_ANGLE, ang, 1000, 90_000, units)
        J, mob = hm.hp_build_read_shockley(1.0, 15.0, 500, 90, 1000, mobility=True)
        lat.hp_set_anisotropy(units, 90_000, 500, J, mob)
        s.update(lat=lat, q=q, m=None, q0=q0, m0=None, keep=units)
    elif kind == "plasticity":
        P = c["points"]
        grain, quat = _plastic_inputs(c, seed)
        s.update(grain=grain, quat=quat, prm=cp_params_table1(1e-4, 7.0), seed=seed, **_cp_state(P),
                 sigma=_f32(6 * P), w=_f32(P), erho=_f32(P))
    elif kind == "train":
        X, Y = _train_data(c, seed)
        s.update(X=X, Y=Y, net=_net(seed))
    elif kind == "elastic":
        grain, quat, epp, E = _elastic_inputs(c, seed)
        n = _sites(c)
        s.update(grain=grain, quat=quat, epp=epp, E=E, prm=cp_params_table1(1e-4, 7.0), eps=_f32(6 * n), sigma=_f32(6 * n))
    else:
        n, G = _sites(c), c["grains"]
        lat = hm.Lattice(c["dim"], (c["x"], c["y"], c["z"])[: c["dim"]], 8 if c["dim"] == 2 else 26, 256, seed, G)
        q, m, quat = _i32(n), _i32(n), _f32(4 * G).view(G, 4)
        pos = torch.empty(G, dtype=torch.int64, device="cuda")
        lat.hp_bind(q, m)
        s.update(lat=lat, q=q, m=m, quat=quat, pos=pos)
    return s


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------
def _restart(v):
    v["lat"].hp_set_spins(v["q0"], v["m0"])
    v["lat"].hp_set_sweep_counter(0)


def _state(v):
    return [v["q"]] if v["m"] is None else [v["q"], v["m"]]


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("sweep", "aniso"):
        _restart(s)
        s["lat"].hp_sweep(c["mcs"])
        return _state(s)
    if kind == "hybrid":
        _restart(s)
        hm.hp_cp_reset(s["prm"], s["q0"].numel(), s["eps"], s["gam"], s["g"])
        hm.hp_cp_step(s["prm"], s["seed"], s["q0"], s["quat"], 0, 2, s["eps"], s["gam"], s["g"], b=s["b"])
        s["lat"].hp_sweep(c["mcs"])
        st, hist = s["lat"].hp_measure(hm.ORIENT_SO3, s["quat"])
        return [*_state(s), s["b"], s["eps"], s["gam"], s["g"], hist, st.alive, st.field_sum, st.mean_mmax]
    if kind == "surrogate":
        _restart(s)
        hm.hp_sur_field(s["net"], s["quat"], c["grains"], s["load"], 7.0, s["b"], s["e"])
        s["lat"].hp_sweep(c["mcs"])
        return [s["q"], s["b"], s["e"]]
    if kind in ("ensemble3d", "ensemble2d"):
        for v in s["members"]:
            _restart(v)
        s["ens"].hp_ensemble_sweep(c["mcs"])
        out = [v["q"] for v in s["members"]]
        if kind == "ensemble2d":
            acc = None
            for v in s["members"]:
                acc = v["lat"].hp_measure(hm.ORIENT_ANGLE, v["orient"], acc=acc)
            out += [acc[1], acc[0].alive, acc[0].field_sum]
        return out
    if kind == "plasticity":
        hm.hp_cp_reset(s["prm"], c["points"], s["eps"], s["gam"], s["g"])
        hm.hp_cp_step(s["prm"], s["seed"], s["grain"], s["quat"], 0, c["incr"], s["eps"], s["gam"], s["g"],
                      sigma=s["sigma"], w=s["w"], erho=s["erho"], b=s["b"])
        return [s["eps"], s["gam"], s["g"], s["sigma"], s["w"], s["erho"], s["b"]]
    if kind == "train":
        p = s["net"].clone()
        m, v, loss = torch.zeros_like(p), torch.zeros_like(p), torch.empty(1, device="cuda")
        hm.hp_sur_train(p, m, v, s["X"], s["Y"], c["steps"], batch=c["batch"], group=GROUP, lr=LR, lr_floor=LR_FLOOR,
                        loss=loss)
        return [p, m, v, loss]
    if kind == "elastic":
        it, _ = hm.hp_elastic_solve(s["prm"], (c["x"], c["y"], c["z"]), s["grain"], s["quat"], s["E"], s["eps"],
                                    eps_p=s["epp"], sigma=s["sigma"], tol=1e-9, max_iter=c["iters"])
        return [s["eps"], s["sigma"], it]
    s["lat"].hp_init_voronoi(hm.ORIENT_SO3, s["quat"], s["pos"])
    return [s["q"], s["m"], s["pos"], s["quat"]]


def work(case):
    """Bytes: a lattice, a point state or a strain field is far larger than what stays on chip
    between two steps (of the small ones it is the same count), so every MCS, refresh and iteration
    reads and writes its state once."""
    c = case
    kind, n = c["kind"], _sites(c) if "x" in c else 0
    if kind == "sweep":     # q (and mp) read and written, the per-point field read
        return {"bytes": n * c["mcs"] * (20 if c["field"] == "point" else 8), "flops": 0}
    if kind == "aniso":
        return {"bytes": 8 * n * c["mcs"], "flops": 0}
    if kind == "hybrid":    # state written once, read and written once, field; then the sweep and the counts
        return {"bytes": n * (32 + 64 + 8 + 20 * c["mcs"] + 12), "flops": 600.0 * 2 * n}
    if kind == "surrogate":
        return {"bytes": 8 * n * c["mcs"] + 24 * c["grains"], "flops": 2.0 * 9024 * c["grains"]}
    if kind == "ensemble3d":
        return {"bytes": 8 * c["mcs"] * sum(m["edge"] ** 3 for m in _members3d(c)), "flops": 0}
    if kind == "ensemble2d":
        return {"bytes": c["replicas"] * n * (8 * c["mcs"] + 4), "flops": 0}
    if kind == "plasticity":
        return {"bytes": c["points"] * (4 + 32 + 32 + 36), "flops": 600.0 * c["points"] * c["incr"]}
    if kind == "train":
        return {"bytes": 52 * c["batch"] * c["steps"], "flops": 6.0 * 9024 * c["batch"] * c["steps"]}
    if kind == "elastic":   # strain read and written, plastic strain and grain read, per iteration; the stress once
        return {"bytes": n * ((48 + 28) * c["iters"] + 24),
                "flops": float(n) * c["iters"] * (2 * 6 * 2.5 * math.log2(max(2, n)) + 400)}
    return {"bytes": 8 * n + 24 * c["grains"], "flops": 0}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------------
def _philox(seed, c0, c2, c3):
    """Words 0..3 of Philox4x32-10 for counters (c0, 0, c2, c3), int64 tensors holding uint32."""
    mask = 0xFFFFFFFF
    c = [c0 & mask, torch.zeros_like(c0), torch.full_like(c0, c2), torch.full_like(c0, c3)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _rotations(quat):
    w, x, y, z = (quat.double() / quat.double().norm(dim=-1, keepdim=True)).unbind(-1)
    r = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(r, dim=-1).reshape(*quat.shape[:-1], 3, 3)


_VI, _VJ = (0, 1, 2, 1, 0, 0), (0, 1, 2, 2, 2, 1)


def _hooke(e, C11, C12, C44):
    """Cubic stress of Voigt rows e[6, ...] (tensor components)."""
    tr = C12 * (e[0] + e[1] + e[2])
    return torch.stack([(C11 - C12) * e[0] + tr, (C11 - C12) * e[1] + tr, (C11 - C12) * e[2] + tr,
                        2 * C44 * e[3], 2 * C44 * e[4], 2 * C44 * e[5]])


def _exact_plasticity(c, seed):
    t1 = synth.TABLE1
    C = (t1["C11"], t1["C12"], t1["C44"])
    tau0, taus, h0, beta = t1["tau0"], t1["taus"], t1["h0"], t1["beta"]
    hr, G = h0 / (taus - tau0), (C[0] - C[1] + 3 * C[2]) / 5
    normals = [(1, 1, 1)] * 3 + [(-1, 1, 1)] * 3 + [(1, -1, 1)] * 3 + [(1, 1, -1)] * 3
    slips = [(0, 1, -1), (-1, 0, 1), (1, -1, 0), (0, 1, -1), (1, 0, 1), (1, 1, 0),
             (0, 1, 1), (1, 0, -1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, -1, 0)]
    nv = torch.tensor(normals, device="cuda", dtype=torch.float64) / math.sqrt(3.0)
    mv = torch.tensor(slips, device="cuda", dtype=torch.float64) / math.sqrt(2.0)
    T = 0.5 * (mv[:, :, None] * nv[:, None, :] + nv[:, :, None] * mv[:, None, :])
    P6 = torch.stack([T[:, i, j] for i, j in zip(_VI, _VJ)], dim=1)          # [12, 6]
    two = torch.tensor([1.0, 1, 1, 2, 2, 2], device="cuda", dtype=torch.float64)
    k = (P6 * two * _hooke(P6.T, *C).T).sum(1)                               # P:C:P
    grain, quat = _plastic_inputs(c, seed)
    out = [[] for _ in range(6)]
    for lo in range(0, c["points"], 1 << 18):
        gr = grain[lo:lo + (1 << 18)].long()
        R = _rotations(quat)[gr]
        load = torch.tensor([1.0, -0.5, -0.5], device="cuda", dtype=torch.float64)
        full = torch.einsum("pki,k,pkj->pij", R, load, R)
        U = torch.stack([full[:, i, j] for i, j in zip(_VI, _VJ)])
        n = gr.numel()
        p = torch.arange(lo, lo + n, device="cuda", dtype=torch.int64)
        ep, gam = torch.zeros(6, n, device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.float64)
        g = torch.full_like(gam, tau0)
        for t in range(1, c["incr"] + 1):
            tau = (P6 * two) @ _hooke(t * 1e-4 * U - ep, *C)                 # [12, n]
            at = tau.abs()
            cand = at > g
            x1 = (at - g) / (k[:, None] + (taus - g) * hr)
            dE = torch.where(cand, -x1 * at + 0.5 * x1 * x1 * k[:, None], torch.full_like(at, math.inf))
            low = dE.min(dim=0).values
            wgt = torch.where(cand, torch.exp(-beta * (dE - torch.where(low.isinf(), torch.zeros_like(low), low))),
                              torch.zeros_like(at))
            cum = wgt.cumsum(0)
            r = _philox(seed, p, t, 1 << 24)[0].double() / 2.0 ** 32
            pick = ((r * cum[-1]) >= cum).sum(0).clamp(max=11)
            last = 11 - cand.flip(0).to(torch.int8).argmax(0)
            pick = torch.minimum(pick, last)
            some = cand.any(0)
            tp = tau.gather(0, pick[None])[0]
            kp, a = k[pick], tp.abs()
            x = (a - g) / (kp + (taus - g) * hr)
            for _ in range(6):
                ey = torch.exp(-hr * x)
                x = x - (a - x * kp - (taus - (taus - g) * ey)) / (-kp - (taus - g) * hr * ey)
            x = torch.where(some, x, torch.zeros_like(x))
            ep = ep + x * torch.sign(tp) * P6[pick].T
            gam = gam + x
            g = torch.where(some, a - kp * x, g)
        ee = c["incr"] * 1e-4 * U - ep
        s = _hooke(ee, *C)
        w = 0.5 * (s * ee * two[:, None]).sum(0)
        for o, v in zip(out, (ep, gam, g, s, w, 2 * g * g / G)):
            o.append(v)
    return [torch.cat(v, dim=-1).reshape(-1) for v in out] + [None]


def _split(p):
    shapes = [(64, 11), (64,), (64, 64), (64,), (64, 64), (64,), (2, 64), (2,)]
    out, at = [], 0
    for sh in shapes:
        n = int(np.prod(sh))
        out.append(p[at:at + n].view(sh))
        at += n
    return out


def _mlp(p, X):
    w = _split(p)
    h = X
    for l in range(3):
        h = torch.nn.functional.gelu(h @ w[2 * l].T + w[2 * l + 1])
    return h @ w[6].T + w[7]


def _exact_train(c, seed):
    X, Y = (v.double() for v in _train_data(c, seed))
    p = _net(seed).double()
    m, v, B = torch.zeros_like(p), torch.zeros_like(p), c["batch"]
    loss = None
    for t in range(1, c["steps"] + 1):
        lo = ((t - 1) % (X.shape[0] // B)) * B
        q = p.clone().requires_grad_(True)
        loss = ((_mlp(q, X[lo:lo + B]) - Y[lo:lo + B]) ** 2).sum() / (2 * B)
        (gr,) = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
        lr = LR * (LR_FLOOR + (1 - LR_FLOOR) * 0.5 * (1 + math.cos(math.pi * t / c["steps"])))
        p = p - lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return [p, m, v, loss.detach().reshape(1)]


def _exact_elastic(c, seed):
    t1 = synth.TABLE1
    C11, C12, C44 = t1["C11"], t1["C12"], t1["C44"]
    grain, quat, epp, E = _elastic_inputs(c, seed)
    n = (c["z"], c["y"], c["x"])
    mu = 0.5 * (C44 + 0.5 * (C11 - C12))
    lam = (C11 + 2 * C12) / 3 - 2 * mu / 3
    Rg = _rotations(quat)

    def stress(eps):
        out = torch.empty_like(eps)
        for lo in range(0, eps.shape[1], 1 << 21):
            sl = slice(lo, lo + (1 << 21))
            R = Rg[grain[sl].long()]
            e = eps[:, sl]
            full = torch.stack([e[0], e[5], e[4], e[5], e[1], e[3], e[4], e[3], e[2]], dim=-1).reshape(-1, 3, 3)
            cr = R.transpose(1, 2) @ full @ R
            ec = torch.stack([cr[:, i, j] for i, j in zip(_VI, _VJ)]) - epp[:, sl].double()
            v = _hooke(ec, C11, C12, C44)
            full = torch.stack([v[0], v[5], v[4], v[5], v[1], v[3], v[4], v[3], v[2]], dim=-1).reshape(-1, 3, 3)
            sm = R @ full @ R.transpose(1, 2)
            out[:, sl] = torch.stack([sm[:, i, j] for i, j in zip(_VI, _VJ)])
        return out

    ks = [torch.fft.fftfreq(v, d=1.0 / v, device="cuda", dtype=torch.float64) for v in n]
    kz, ky, kx = torch.meshgrid(*ks, indexing="ij")
    nyq = torch.zeros(n, dtype=torch.bool, device="cuda")
    for k, v in zip((kz, ky, kx), n):
        if v % 2 == 0:
            nyq |= k == -v // 2
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    nv = [k / k2.sqrt() for k in (kx, ky, kz)]
    kap = (lam + mu) / (mu * (lam + 2 * mu))
    eps = torch.tensor(E, device="cuda", dtype=torch.float64)[:, None].repeat(1, _sites(c))
    for _ in range(c["iters"]):
        tau = stress(eps) - 2 * mu * eps
        tau[:3] -= lam * (eps[0] + eps[1] + eps[2])
        th = [torch.fft.fftn(tau[i].reshape(n)) for i in range(6)]
        a = [th[0] * nv[0] + th[5] * nv[1] + th[4] * nv[2], th[5] * nv[0] + th[1] * nv[1] + th[3] * nv[2],
             th[4] * nv[0] + th[3] * nv[1] + th[2] * nv[2]]
        cc = a[0] * nv[0] + a[1] * nv[1] + a[2] * nv[2]
        for i, (p, q) in enumerate(zip(_VI, _VJ)):
            o = -((nv[p] * a[q] + a[p] * nv[q]) * (0.5 / mu) - kap * cc * nv[p] * nv[q])
            o[nyq] = 0
            o[0, 0, 0] = E[i] * _sites(c)
            eps[i] = torch.fft.ifftn(o).real.reshape(-1)
    return [eps.reshape(-1), stress(eps).reshape(-1), None]


def _exact_quats(G, seed):
    u = [w.double() / 2.0 ** 32 for w in _philox(seed, torch.arange(G, device="cuda", dtype=torch.int64), 0, (2 << 24) | 1)]
    a, b = (1 - u[0]).sqrt(), u[0].sqrt()
    return torch.stack([a * torch.sin(2 * math.pi * u[1]), a * torch.cos(2 * math.pi * u[1]),
                        b * torch.sin(2 * math.pi * u[2]), b * torch.cos(2 * math.pi * u[2])], dim=1)


def exact(case, seed):
    """Lattices, ids, counts and quantised fields are whole numbers: only the computed reals here."""
    c, seed = dict(case), int(seed)
    kind = c["kind"]
    if kind == "plasticity":
        return _exact_plasticity(c, seed)
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "elastic":
        return _exact_elastic(c, seed)
    if kind == "voronoi":
        return [None, None, None, _exact_quats(c["grains"], seed)]
    if kind == "surrogate":
        R = _rotations(_exact_quats(c["grains"], seed).float())
        d = R[:, 0, :].abs().sort(dim=1, descending=True).values
        inv = (d[:, 0] * d[:, 1]) ** 2 + (d[:, 1] * d[:, 2]) ** 2 + (d[:, 2] * d[:, 0]) ** 2
        load = torch.tensor([0.55, -0.27, -0.28, 0.01, -0.02, 0.005, 2.5], device="cuda", dtype=torch.float64)
        X = torch.cat([d, inv[:, None], load.expand(d.shape[0], 7)], dim=1)
        y = _mlp(_net(seed).double(), X)
        return [None, None, 7.0 * (y[:, 0] * 0.01 + y[:, 1] * 0.002)]
    return None

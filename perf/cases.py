"""The measured workloads: control solves through the package's public entry
points, from the smallest to the largest that the configurations, tests and
benchmark of this repository use, with every option that a planner switches
on in earnest.

A scene is a drive along a reference path of a straight and an arc (or of
several, for the long path), forward or in reverse, with obstacles parked
beside it, the vehicle a few centimetres off the path and a nominal input
sequence as a running controller has it (the progress rate about the speed).
Everything is drawn from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2508_05773_gb300 as pkg
from paper_2508_05773_gb300 import scenarios as sc

#: options of a solve -> parameter overrides
OPTIONS = {
    "": {},
    # pedestrians that walk and parked vehicles as super-ellipses (e = 4)
    "moving": {"flags": sc.FLAG_OBS8},
    # three discs on the tractor, two on the trailer, per obstacle
    "moving discs": {"flags": sc.FLAG_OBS8, **sc.FIVE_DISCS},
    # the paper's jerk-input model with third-order obstacle rows
    "moving third jerk": {"flags": sc.FLAG_OBS8 | sc.FLAG_THIRD_ORDER | sc.FLAG_JERK},
    # the comparison method: no projection, a collision cost
    "mppi collision": {"flags": sc.FLAG_PROJ_NONE | sc.FLAG_COLLISION_COST},
}


def listed():
    return [
        # the smallest scene of the configurations: a parking aid's tick, all latency
        {"name": "small solve", "kind": "solve", "options": "", "S": 256, "H": 30, "obstacles": 1, "rows": 389},
        # the paper-scale control tick on device buffers, the benchmark's own size
        {"name": "control solve", "kind": "solve", "options": "", "S": 4096, "H": 50, "obstacles": 8, "rows": 388},
        # the same tick as a closed loop calls it, from host buffers and back
        {"name": "host control solve", "kind": "host", "options": "", "S": 4096, "H": 50, "obstacles": 8, "rows": 388},
        # the paper's own horizon (Table I): ragged sample count, 6 s ahead
        {"name": "long horizon", "kind": "solve", "options": "", "S": 5000, "H": 120, "obstacles": 8, "rows": 388},
        # standard MPPI with a collision cost, the method that Table I compares with
        {"name": "mppi collision", "kind": "solve", "options": "mppi collision", "S": 5000, "H": 120, "obstacles": 8,
         "rows": 388},
        # parked vehicles and crossing pedestrians
        {"name": "crossing", "kind": "solve", "options": "moving", "S": 4096, "H": 50, "obstacles": 8, "rows": 388},
        # the same scene seen from a footprint of five discs: 40 rows a step
        {"name": "crossing five discs", "kind": "solve", "options": "moving discs", "S": 4096, "H": 50,
         "obstacles": 8, "rows": 388},
        # the paper's vehicle model (jerk input) with third-order rows, an odd size
        {"name": "jerk third order", "kind": "solve", "options": "moving third jerk", "S": 3001, "H": 61,
         "obstacles": 7, "rows": 301},
        # a lot full of parked vehicles, many samples: the largest single solve
        {"name": "dense lot", "kind": "solve", "options": "", "S": 65536, "H": 100, "obstacles": 64, "rows": 2401},
        # one tick of a small fleet: as many vehicles as a served batch has
        {"name": "fleet batch", "kind": "batch", "options": "", "instances": 48, "uneven": False, "S": 4096, "H": 50,
         "obstacles": 8, "rows": 388},
        # many vehicles with different sample counts, horizons and obstacles
        {"name": "uneven batch", "kind": "batch", "options": "", "instances": 256, "uneven": True, "S": 8192, "H": 80,
         "obstacles": 16, "rows": 501},
        # the hitch-angle stabilizer over a table of states
        {"name": "stabilize states", "kind": "stabilize", "options": "", "states": 4000001},
    ]


def _cost(case) -> float:
    if case["kind"] == "stabilize":
        return 100.0 * case["states"]
    n = sum(s * h * _ops(o, case["options"]) for s, h, o in _sizes(case))
    return float(n)


def draw(rng: random.Random):
    def spread(lo, hi):  # whole numbers, even over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("solve", "solve", "solve", "solve", "host", "batch", "batch", "stabilize"))
        if kind == "stabilize":
            case = {"kind": kind, "options": "", "states": spread(1, 8000000)}
        elif kind == "batch":
            case = {"kind": kind, "options": "", "instances": spread(1, 256), "uneven": rng.random() < 0.5,
                    "S": spread(256, 8192), "H": rng.randint(20, 80), "obstacles": rng.randint(0, 16),
                    "rows": spread(100, 600)}
        else:
            options = rng.choice(("", "", "", "moving", "moving discs", "moving third jerk", "mppi collision"))
            case = {"kind": kind, "options": options, "S": spread(64, 65536), "H": spread(10, 120),
                    "obstacles": rng.randint(0, 16) if options or rng.random() < 0.6 else spread(16, 64),
                    "rows": spread(100, 2401)}
            if options == "moving discs":
                case["obstacles"] = max(1, case["obstacles"])
        if _cost(case) <= most:
            return case


# ------------------------------------------------------------------- inputs
def _sizes(case):
    """(S, H, obstacles) of every solve of a case."""
    if case["kind"] != "batch":
        return [(case["S"], case["H"], case["obstacles"])]
    if not case["uneven"]:
        return [(case["S"], case["H"], case["obstacles"])] * case["instances"]
    r = random.Random(case["instances"])
    return [(max(1, case["S"] >> r.randrange(4)), r.randint(max(1, 3 * case["H"] // 8), case["H"]),
             r.randint(0, case["obstacles"])) for _ in range(case["instances"])]


def _params(case, S, H):
    return sc.params(S=S, H=H, **OPTIONS[case["options"]])


def _path(rng, rows):
    """A reference path of `rows` rows and the side it is driven on."""
    ds = 0.1 if rows <= 1000 else 0.05
    length = (rows - 1) * ds
    reverse = bool(rng.random() < 0.5)
    segs, total = [], 0.0
    while total < length + 1.0:
        straight = float(rng.uniform(8.0, 15.0))
        R, ang = float(rng.uniform(10.0, 15.0)), float(rng.uniform(0.7, 1.5)) * float(rng.choice((-1.0, 1.0)))
        segs += [("S", straight), ("A", R, ang)]
        total += straight + R * abs(ang)
    return sc.path_table(segs, ds, reverse)[:rows].copy(), ds, reverse


def _scene(case, S, H, n_obs, rng):
    """One solve's host inputs."""
    flags = int(OPTIONS[case["options"]].get("flags", 0))
    path, ds, reverse = _path(rng, case["rows"])
    v0 = float(rng.uniform(0.8, 1.4)) * (-1.0 if reverse else 1.0)
    head = math.pi if reverse else 0.0
    x0 = [float(rng.uniform(-0.05, 0.05)), float(rng.uniform(-0.05, 0.05)), head + float(rng.uniform(-0.02, 0.02)),
          head + float(rng.uniform(-0.04, 0.04)), v0, float(rng.uniform(-0.03, 0.03)), 0.0]
    if flags & sc.FLAG_JERK:
        x0.append(float(rng.uniform(-0.1, 0.1)))
    # obstacles beside the path, most of them along the part that is driven now
    keep = 5.0 if "discs" in case["options"] else 2.6
    obs = []
    for i in range(n_obs):
        ahead = float(rng.uniform(0.0, min(1.0, 25.0 / ((case["rows"] - 1) * ds)) if i % 4 else 1.0))
        x, y, th = (float(v) for v in path[int(ahead * (case["rows"] - 1))])
        side = float(rng.choice((-1.0, 1.0)))
        lat = side * float(rng.uniform(keep, keep + 4.0))
        c = (x - lat * math.sin(th), y + lat * math.cos(th))
        row = [c[0], c[1], float(rng.uniform(0.4, 1.5)), float(rng.uniform(0.3, 0.9)), th + float(rng.uniform(-0.3, 0.3)),
               2.0]
        if flags & sc.FLAG_OBS8:
            if rng.random() < 0.7:  # a parked vehicle
                row[5] = 4.0
                row += [0.0, 0.0]
            else:  # a pedestrian that walks beside or away from the path
                row[2] = row[3] = 0.5
                a, sp = float(rng.uniform(-0.6, 0.6)), side * float(rng.uniform(0.3, 1.2))
                row += [-sp * math.sin(th + a), sp * math.cos(th + a)]
        obs.append(row)
    U = np.empty((H, 3), np.float32)
    t = np.arange(H) * 0.05
    for j, (mean, amp) in enumerate(((0.0, 0.1), (0.0, 0.05), (abs(v0), 0.1))):
        U[:, j] = mean + amp * np.sin(float(rng.uniform(0.3, 2.0)) * t + float(rng.uniform(0.0, 6.0)))
    return dict(x0=np.asarray(x0, np.float64), U_nom=U,
                obs=np.asarray(obs, np.float32).reshape(n_obs, 8 if flags & sc.FLAG_OBS8 else 6), path=path, ds=ds,
                seed=int(rng.integers(0, 2**63 - 1)), counter=int(rng.integers(0, 2**20)), S=S, H=H)


def _scenes(case, seed):
    rng = np.random.default_rng(seed)
    return [_scene(case, S, H, n, rng) for S, H, n in _sizes(case)]


def _states(case, seed):
    """States and reference inputs of the stabilizer, on the GPU: speeds both
    ways, hitch angles up to beyond the limit."""
    n = case["states"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.empty((n, 7), dtype=torch.float64, device="cuda").uniform_(-1.0, 1.0, generator=g)
    x *= torch.tensor([50.0, 50.0, 3.0, 3.0, 3.0, 0.5, 100.0], dtype=torch.float64, device="cuda")
    x[:, 3] = x[:, 2] + x[:, 3] / 3.0
    u = torch.empty((n, 3), dtype=torch.float32, device="cuda").uniform_(-1.0, 1.0, generator=g)
    u *= torch.tensor([2.0, 0.6, 1.5], device="cuda")
    return x, u


def prepare(case, seed):
    if case["kind"] == "stabilize":
        x, u = _states(case, seed)
        solver = pkg.Solver(sc.params(S=64, H=10), max_obstacles=1, max_path_pts=16)
        return dict(kind="stabilize", solver=solver, x=x, u=u, out=torch.empty((case["states"], 4), device="cuda"))
    scenes = _scenes(case, seed)
    S, H = max(s["S"] for s in scenes), max(s["H"] for s in scenes)
    n_obs = max(len(s["obs"]) for s in scenes)
    solver = pkg.Solver(_params(case, S, H), max_obstacles=max(1, n_obs), max_path_pts=case["rows"],
                        max_batch=len(scenes) if case["kind"] == "batch" else 0)
    if case["kind"] == "host":
        return dict(kind="host", solver=solver, scene=scenes[0])
    # outputs side by side, one tensor a kind
    total_h = sum(s["H"] for s in scenes)
    out = dict(U=torch.zeros((total_h, 3), device="cuda"), U_next=torch.zeros((total_h, 3), device="cuda"),
               traj=torch.zeros((total_h + len(scenes), 7), device="cuda"),
               J=torch.zeros(sum(s["S"] for s in scenes), device="cuda"),
               status=torch.full((len(scenes),), 99, dtype=torch.int32, device="cuda"))
    insts, h0, s0 = [], 0, 0
    for i, s in enumerate(scenes):
        dev = {k: torch.as_tensor(s[k], device="cuda") for k in ("x0", "U_nom", "obs", "path")}
        if not len(s["obs"]):
            dev["obs"] = None
        insts.append(dict(dev, ds=s["ds"], S=s["S"], seed=s["seed"], counter=s["counter"],
                          U_out=out["U"][h0:h0 + s["H"]], U_next=out["U_next"][h0:h0 + s["H"]],
                          traj_out=out["traj"][h0 + i:h0 + i + s["H"] + 1], J_out=out["J"][s0:s0 + s["S"]],
                          status=out["status"][i:i + 1]))
        h0, s0 = h0 + s["H"], s0 + s["S"]
    state = dict(kind=case["kind"], solver=solver, insts=insts, out=out)
    if case["kind"] == "batch":
        state["array"] = pkg.make_instances(insts)
    return state


def run(state):
    solver = state["solver"]
    if state["kind"] == "stabilize":
        solver.hitch_stabilize_device(state["x"], state["u"], state["out"])
        return state["out"]
    if state["kind"] == "host":
        s = state["scene"]
        r = solver.solve(s["x0"], s["U_nom"], s["obs"], s["path"], s["ds"], s["seed"], s["counter"])
        return dict(U=r["U"], traj=r["traj"])
    if state["kind"] == "batch":
        solver.solve_batch(state["array"])
        return state["out"]
    d = state["insts"][0]
    rc = solver.solve_device(d["x0"], d["U_nom"], d["obs"], d["path"], d["ds"], d["seed"], d["counter"], d["U_out"],
                             d["traj_out"], d["J_out"], d["U_next"], d["status"])
    if rc != 0:
        raise RuntimeError(pkg.brmppi_last_error(solver.ctx))
    return state["out"]


# --------------------------------------------------------------------- work
def _ops(n_obs, options):
    """Arithmetic operations of one sample's step: a Philox block and its four
    normals 124, the step without rows 115, the hitch row 51, an obstacle
    row 35 (with the steer-rate column and a moving centre about 90)."""
    if "mppi" in options:
        return 124 + 92 + 25 * n_obs
    rows = n_obs * (5 if "discs" in options else 1)
    blocks = (4 + rows + 3) // 4
    return 124 * blocks + 115 + 51 + (90 if options else 35) * rows


def work(case):
    if case["kind"] == "stabilize":
        return {"bytes": 84 * case["states"], "flops": 100 * case["states"]}
    nbytes = 0
    for S, H, n in _sizes(case):
        nbytes += 64 + 12 * H + 32 * n + 12 * case["rows"] + 12 * H + 28 * (H + 1)
        if case["kind"] != "host":
            nbytes += 4 * S + 12 * H + 4
    return {"bytes": nbytes, "flops": _cost(case)}


# -------------------------------------------------------------------- exact
_D = torch.float64


def _philox(b, tau, s, ctr, key0, key1):
    """Philox4x32-10 words (Salmon et al., SC'11) in 64-bit integers."""
    m = 0xFFFFFFFF
    c = [b, tau, s, ctr]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # modulo 2^64
        c = [((p1 >> 32) & m) ^ c[1] ^ key0, p1 & m, ((p0 >> 32) & m) ^ c[3] ^ key1, p0 & m]
        key0, key1 = (key0 + 0x9E3779B9) & m, (key1 + 0xBB67AE85) & m
    return c


def _normals(n, tau, S, ctr, key0, key1):
    """Normals 0..n-1 of step tau, (B, n, S); ctr and keys (B,)."""
    blocks = (n + 3) // 4
    dev = ctr.device
    b = torch.arange(blocks, device=dev)[None, :, None]
    s = torch.arange(S, device=dev)[None, None, :]
    one = torch.zeros((len(ctr), blocks, S), dtype=torch.int64, device=dev)
    col = lambda v: v[:, None, None]  # noqa: E731
    w = _philox(one + b, one + tau, one + s, one + col(ctr), one + col(key0), one + col(key1))
    u = [((x >> 9).to(_D) + 0.5) * 2.0**-23 for x in w]
    out = torch.empty((len(ctr), blocks, 4, S), dtype=_D, device=dev)
    for j in (0, 2):
        r = torch.sqrt(-2.0 * torch.log(u[j]))
        out[:, :, j] = r * torch.cos(2.0 * math.pi * u[j + 1])
        out[:, :, j + 1] = r * torch.sin(2.0 * math.pi * u[j + 1])
    return out.reshape(len(ctr), 4 * blocks, S)[:, :n]


def _wrap(a):
    return a - 2.0 * math.pi * torch.round(a / (2.0 * math.pi))


def _exact_solves(scenes, p, flags):
    """U*, trajectory and costs of solves of the same parameters in 64 bits
    (padded to the largest of them): rollouts, softmin and update, by the
    definitions of the paper (rows through hdot and hddot, the projection by
    its Woodbury form)."""
    dev = "cuda"
    t = lambda a, dt=_D: torch.as_tensor(np.asarray(a), device=dev).to(dt)  # noqa: E731
    B, S, H = len(scenes), max(s["S"] for s in scenes), max(s["H"] for s in scenes)
    N = max(len(s["obs"]) for s in scenes)
    n_pts = max(len(s["path"]) for s in scenes)
    pad = lambda a, n: np.concatenate([a, np.repeat(a[-1:], n - len(a), axis=0)]) if len(a) < n else a  # noqa: E731
    x0 = t(np.stack([s["x0"] for s in scenes]))
    Unom = t(np.stack([pad(s["U_nom"], H) for s in scenes]))
    path = t(np.stack([pad(s["path"], n_pts) for s in scenes]))
    Sb, Hb = t([s["S"] for s in scenes], torch.int64), t([s["H"] for s in scenes], torch.int64)
    ds = t(np.float32(scenes[0]["ds"]))
    far = np.array([[1e3, 1e3, 1.0, 1.0, 0.0, 2.0, 0.0, 0.0]])
    obs = t(np.stack([np.concatenate([np.pad(s["obs"].astype(np.float64), ((0, 0), (0, 8 - s["obs"].shape[1]))),
                                      np.repeat(far, N - len(s["obs"]), axis=0)]) for s in scenes]))
    live = t(np.stack([np.arange(N) < len(s["obs"]) for s in scenes]))
    proj, jerk, third = not flags & sc.FLAG_PROJ_NONE, bool(flags & sc.FLAG_JERK), bool(flags & sc.FLAG_THIRD_ORDER)
    nd = int(p["n_discs"])
    key0, key1 = (t([(s["seed"] >> sh) & 0xFFFFFFFF for s in scenes], torch.int64) for sh in (0, 32))
    ctr = t([s["counter"] & 0xFFFFFFFF for s in scenes], torch.int64)
    Ts, l1, l2, lh = p["Ts"], p["l1"], p["l2"], p["lh"]
    kh = lh / l1
    zlo, zhi = p["z_lo"], p["z_hi"]
    st = lambda j: x0[:, j, None].expand(B, S).clone()  # noqa: E731
    px, py, th1, th2, v, dl, psi = (st(j) for j in range(7))
    acc = st(7) if jerk else torch.zeros_like(px)
    m_a = p["w_alpha"] + p["rho"]
    m_u = [p["w_u"][j] + p["rho"] for j in range(3)]
    alpha = torch.full((B, 1 + N * nd, S), p["alpha0"], dtype=_D, device=dev)
    live_row = live.repeat_interleave(nd, dim=1)[:, :, None]
    J = torch.zeros((B, S), dtype=_D, device=dev)
    hist = torch.empty((H, 3, B, S), dtype=torch.float64, device=dev)
    o = lambda j: obs[:, :, j, None]  # noqa: E731  (B, N, 1)
    co, so = torch.cos(o(4)), torch.sin(o(4))
    e4 = o(5) == 4.0
    Ax, Ay = o(2) + p["r_inflate"], o(3) + p["r_inflate"]

    def ellipse(xp, yp):
        """h and its derivatives along the axes: value, (hx, hy), (hxx, hyy), (hxxx, hyyy)."""
        X, Y = torch.where(e4, xp**2 / Ax**4, 1 / Ax**2), torch.where(e4, yp**2 / Ay**4, 1 / Ay**2)
        c1, c2 = torch.where(e4, 4.0, 2.0).to(_D), torch.where(e4, 12.0, 2.0).to(_D)
        third_ = (torch.where(e4, 24 * xp / Ax**4, 0.0), torch.where(e4, 24 * yp / Ay**4, 0.0))
        return xp**2 * X + yp**2 * Y - 1, (c1 * xp * X, c1 * yp * Y), (c2 * X, c2 * Y), third_

    def rot(wx, wy):
        return co * wx + so * wy, co * wy - so * wx

    def disc(m):
        tr = (int(p["disc_trailer_mask"]) >> m) & 1
        return (-lh, -(l2 - p["disc_off"][m])) if tr else (p["disc_off"][m], 0.0)

    for tau in range(H):
        noise = _normals(4 + N * nd if proj else 3, tau, S, ctr, key0, key1)
        zd = [torch.clamp(Unom[:, tau, j, None] + p["sigma"][j] * noise[:, j], zlo[j], zhi[j]) for j in range(3)]
        c1, s1, c2, s2 = torch.cos(th1), torch.sin(th1), torch.cos(th2), torch.sin(th2)
        tn, phi = torch.tan(dl), th1 - th2
        sp, cp = torch.sin(phi), torch.cos(phi)
        sec2, G = 1 + tn**2, sp - kh * cp * tn
        w1, w2 = v * tn / l1, v * G / l2  # heading rates
        if proj:
            zda = torch.clamp(p["sigma_alpha"] * noise[:, 3:], p["ua_lo"], p["ua_hi"])
            pam = (p["w_alpha"] * zda + 0.5 * p["rho"] * (p["ua_hi"] + p["ua_lo"])) / m_a
            # heading accelerations: constant, per a, per omega
            a1a, a1w = tn / l1, v * sec2 / l1
            a20 = v / l2 * (cp + kh * tn * sp) * (w1 - w2)
            a2a, a2w = G / l2, -v / l2 * kh * cp * sec2
            sg = torch.where(th2 - th1 >= 0, 1.0, -1.0).to(_D)
            hh = p["dtheta_max"] - p["kappa"] * v - (th2 - th1).abs()
            half = 0.5 * Ts * Ts
            Aa, Aw = -Ts * p["kappa"] - half * sg * (a2a - a1a), -half * sg * (a2w - a1w)
            cc = -Ts * sg * (w2 - w1) - half * sg * a20
            if jerk:
                cc, Aa = cc + acc * Aa, torch.full_like(Aa, -half * p["kappa"])
            hs, As, Ws, Cs = [hh[:, None]], [Aa[:, None]], [Aw[:, None]], [cc[:, None]]
            if N:
                q = lambda a: a[:, None, :]  # noqa: E731
                rows = []
                for m in range(nd):
                    d1, d2 = disc(m)
                    pxm = px + d1 * c1 + d2 * c2
                    pym = py + d1 * s1 + d2 * s2
                    time = tau * Ts
                    xp, yp = rot(q(pxm) - (o(0) + time * o(6)), q(pym) - (o(1) + time * o(7)))
                    h, g, hs2, hs3 = ellipse(xp, yp)
                    vel = rot(q(v * c1 - d1 * w1 * s1 - d2 * w2 * s2) - o(6), q(v * s1 + d1 * w1 * c1 + d2 * w2 * c2) - o(7))
                    ac0 = rot(q(-v * w1 * s1 - d1 * w1**2 * c1 - d2 * (a20 * s2 + w2**2 * c2)),
                              q(v * w1 * c1 - d1 * w1**2 * s1 + d2 * (a20 * c2 - w2**2 * s2)))
                    aca = rot(q(c1 - d1 * a1a * s1 - d2 * a2a * s2), q(s1 + d1 * a1a * c1 + d2 * a2a * c2))
                    acw = rot(q(-d1 * a1w * s1 - d2 * a2w * s2), q(d1 * a1w * c1 + d2 * a2w * c2))
                    dot = lambda a, b: a[0] * b[0] + a[1] * b[1]  # noqa: E731
                    const = Ts * dot(g, vel) + half * (dot(g, ac0) + hs2[0] * vel[0]**2 + hs2[1] * vel[1]**2)
                    ra, rw = half * dot(g, aca), half * dot(g, acw)
                    if third:
                        n1 = rot(q(-s1), q(c1))
                        e1 = rot(q(c1), q(s1))
                        Hw = (hs2[0] * vel[0], hs2[1] * vel[1])
                        s3 = Ts**3 / 6
                        ra = ra + s3 * (dot(g, n1) * q(2 * w1 + v * a1a) + 3 * dot(Hw, e1))
                        rw = rw + s3 * dot(g, n1) * q(v * a1w)
                        const = const + s3 * (-q(v * w1**2) * dot(g, e1) + 3 * q(v * w1) * dot(Hw, n1) +
                                              hs3[0] * vel[0]**3 + hs3[1] * vel[1]**3)
                        if jerk:
                            const, ra = const + q(acc) * ra, s3 * dot(g, e1).expand_as(ra)
                    elif jerk:
                        const, ra = const + q(acc) * ra, torch.zeros_like(ra)
                    rows.append((h, ra, rw, const))
                pack = [torch.stack([r[k].expand(B, N, S) for r in rows], dim=2).reshape(B, N * nd, S) for k in range(4)]
                for to, x in zip((hs, As, Ws, Cs), pack):
                    to.append(x)
            h, A, W, C = (torch.cat(x, dim=1) for x in (hs, As, Ws, Cs))
            keep = torch.cat([torch.ones((B, 1, 1), dtype=_D, device=dev), live_row], dim=1)
            hm = torch.clamp(h.abs(), min=p["h_floor"])
            ht = torch.where(h >= 0, hm, -hm)
            pu = [(p["w_u"][j] * zd[j] + 0.5 * p["rho"] * (zhi[j] + zlo[j])) / m_u[j] for j in range(3)]
            r = A * pu[0][:, None] + W * pu[1][:, None] + ht * pam + alpha * h + C
            ua, uw, rho = keep * A / ht, keep * W / ht, r / ht
            S00, S01, S11 = m_u[0] + m_a * (ua * ua).sum(1), m_a * (ua * uw).sum(1), m_u[1] + m_a * (uw * uw).sum(1)
            g0, g1 = m_a * (ua * rho).sum(1), m_a * (uw * rho).sum(1)
            det = S00 * S11 - S01 * S01
            y0, y1 = (S11 * g0 - S01 * g1) / det, (S00 * g1 - S01 * g0) / det
            z = [pu[0] - y0, pu[1] - y1, pu[2]]
            alpha = alpha + pam - rho + ua * y0[:, None] + uw * y1[:, None]
        else:
            z = zd
        u = [torch.clamp(z[j], zlo[j], zhi[j]) for j in range(3)]
        hist[tau] = torch.stack(u)
        px, py, th1, th2 = px + Ts * v * c1, py + Ts * v * s1, th1 + Ts * w1, th2 + Ts * w2
        if jerk:
            v, acc = v + Ts * acc, acc + Ts * u[0]
        else:
            v = v + Ts * u[0]
        dl, psi = dl + Ts * u[1], psi + Ts * u[2]
        # stage cost at the new state
        last = t([len(s["path"]) - 1 for s in scenes])[:, None]
        f = torch.minimum(torch.clamp(psi / ds, min=0.0), last)
        i = torch.minimum(torch.floor(f), last - 1)
        f, i = f - i, i.to(torch.int64)
        row = lambda k, j: torch.gather(path[:, :, j], 1, i + k)  # noqa: E731
        xr, yr, thr = (row(0, j) + f * (row(1, j) - row(0, j)) for j in range(3))
        ec = torch.sin(thr) * (px - xr) - torch.cos(thr) * (py - yr)
        el = -torch.cos(thr) * (px - xr) - torch.sin(thr) * (py - yr)
        cost = p["Qc"] * ec**2 + p["Ql"] * el**2 + p["Qth"] * (_wrap(th1 - thr)**2 + _wrap(th2 - thr)**2)
        cost = cost + sum(p["R"][j] * u[j]**2 for j in range(3)) + p["mu"] * (p["nu_bar"] - u[2])**2
        if flags & sc.FLAG_COLLISION_COST and N:
            time = (tau + 1) * Ts
            h = ellipse(*rot(px[:, None] - (o(0) + time * o(6)), py[:, None] - (o(1) + time * o(7))))[0]
            cost = cost + p["q_coll"] * (live_row * torch.clamp(-h, min=0.0)).sum(1)
        J = J + torch.where((tau < Hb)[:, None], cost, 0.0)
    real = torch.arange(S, device=dev)[None] < Sb[:, None]
    J = torch.where(real, J, math.inf)
    w = torch.softmax(-J / p["lambda"], dim=1)
    U = (hist * w[None, None]).sum(3).permute(2, 0, 1)  # (B, H, 3)
    out = []
    for b, s in enumerate(scenes):
        Ub = U[b, :s["H"]]
        x = [float(a) for a in s["x0"]]
        traj = [x[:7]]
        for a, om, nu in Ub.tolist():
            tq = math.tan(x[5])
            ph = x[2] - x[3]
            nx = [x[0] + Ts * x[4] * math.cos(x[2]), x[1] + Ts * x[4] * math.sin(x[2]), x[2] + Ts * x[4] * tq / l1,
                  x[3] + Ts * x[4] / l2 * (math.sin(ph) - kh * math.cos(ph) * tq),
                  x[4] + Ts * (x[7] if jerk else a), x[5] + Ts * om, x[6] + Ts * nu]
            x = nx + ([x[7] + Ts * a] if jerk else [])
            traj.append(x[:7])
        out.append((Ub, torch.tensor(traj, dtype=_D, device=dev), J[b, :s["S"]]))
    return out


def _exact_stabilizer(case, seed, p):
    """The one-row QP with a box in 64 bits: the multiplier by its breakpoints."""
    x, u = _states(case, seed)
    u = u.to(_D)
    Ts, kh = p["Ts"], p["lh"] / p["l1"]
    v, tn, phi = x[:, 4], torch.tan(x[:, 5]), x[:, 2] - x[:, 3]
    sp, cp, sec2 = torch.sin(phi), torch.cos(phi), 1 + tn**2
    G = sp - kh * cp * tn
    w1, w2 = v * tn / p["l1"], v * G / p["l2"]
    sg = torch.where(phi <= 0, 1.0, -1.0).to(_D)
    half = 0.5 * Ts * Ts
    g = torch.stack([-Ts * p["kappa"] - half * sg * (G / p["l2"] - tn / p["l1"]),
                     half * sg * v * sec2 * (kh * cp / p["l2"] + 1 / p["l1"])], 1)
    c0 = -Ts * sg * (w2 - w1) - half * sg * v / p["l2"] * (cp + kh * tn * sp) * (w1 - w2)
    rhs = -p["alpha_stab"] * (p["dtheta_max"] - p["kappa"] * v - phi.abs()) - c0
    lo, hi = (torch.tensor(p[k][:2], dtype=_D, device=x.device) for k in ("z_lo", "z_hi"))
    d = g / torch.tensor(p["q_stab"], dtype=_D, device=x.device)
    ref = u[:, :2]
    at = lambda mu: torch.minimum(torch.maximum(ref + mu[:, None] * d, lo), hi)  # noqa: E731
    breaks = torch.cat([(lo - ref) / d, (hi - ref) / d], 1)
    breaks = torch.where((breaks > 0) & torch.isfinite(breaks), breaks, math.inf).sort(1).values
    mu, f = torch.zeros_like(v), (g * at(torch.zeros_like(v))).sum(1)
    best, done = torch.zeros_like(v), f >= rhs
    for k in range(4):
        m = breaks[:, k]
        ok = torch.isfinite(m)
        m1 = torch.where(ok, m, mu)
        f1 = (g * at(m1)).sum(1)
        hit = ok & ~done & (f1 >= rhs)
        best = torch.where(hit, mu + (rhs - f) * (m1 - mu) / (f1 - f), best)
        done = done | hit
        mu, f = m1, f1
    corner = torch.where(d > 0, hi, torch.where(d < 0, lo, at(torch.zeros_like(v))))
    a = torch.where(done[:, None], at(best), corner)
    return torch.cat([a, u[:, 2:], ((g * a).sum(1) - rhs)[:, None]], 1)


def exact(case, seed):
    p = sc.as_float32(sc.params(**OPTIONS[case["options"]]))
    if case["kind"] == "stabilize":
        return _exact_stabilizer(case, seed, p)
    scenes = _scenes(case, seed)
    solved = [None] * len(scenes)
    # solves of about the same size together, as many as fit about 2 GB of rows
    order = sorted(range(len(scenes)), key=lambda i: (scenes[i]["S"], scenes[i]["H"]))
    while order:
        size = lambda g: len(g) * max((len(scenes[i]["obs"]) * int(p["n_discs"]) + 4) * scenes[i]["S"] for i in g)  # noqa: E731
        group = [order.pop()]
        while order and size(group + order[-1:]) < 6e6:
            group.append(order.pop())
        for i, r in zip(group, _exact_solves([scenes[i] for i in group], p, int(p["flags"]))):
            solved[i] = r
    U, traj, J = (torch.cat([s[k] for s in solved]) for k in range(3))
    if case["kind"] == "host":
        return dict(U=U, traj=traj)
    U_next = torch.cat([torch.cat([s[0][1:], s[0][-1:]]) for s in solved])
    return dict(U=U, U_next=U_next, traj=traj, J=J, status=None)

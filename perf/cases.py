"""The calls that programs built on this library make, as measurable cases.

A case names a scene (a generator of ``paper_2005_06773_gb300.scenarios`` with its sizes), a call (the public entry
point that takes the scene) and whether the caller brings its own trajectory weights.  ``listed()`` is the fixed
list, ``draw()`` gives further cases of the same ranges, ``prepare()`` makes what a program holds before the call,
``run()`` makes the call, ``work()`` says what it cannot do without and ``exact()`` gives its floating outputs in
64 bits, from the model equations alone.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2005_06773_gb300 import mhc
from paper_2005_06773_gb300 import scenarios as S

# ---------------------------------------------------------------------------------------------------------
# the cases


def _case(name, call, scene, n_acc, n_str, n_steps, n_ped_v=0, n_ped_h=0, count=1, sizes=3, weighted=False):
    return dict(name=name, call=call, scene=scene, n_acc=n_acc, n_str=n_str, n_steps=n_steps, n_ped_v=n_ped_v,
                n_ped_h=n_ped_h, count=count, sizes=sizes, weighted=weighted)


def listed():
    return [
        # two cars at a crossing from host inputs to host outputs: the smallest request, all latency
        _case("crossing_run", "run", "crossing", 4, 4, 20),
        # the 11-object intersection, everything resident on the device: the latency of one sensor frame
        _case("intersection_evaluate", "evaluate", "intersection", 21, 21, 30, 11, 11),
        # the same from host inputs and the caller's own weights to host outputs: the call of a controller
        _case("intersection_run", "run", "intersection", 21, 21, 30, 11, 11, weighted=True),
        # a stream of sensor frames of one structure: a plan, updated with the frame's states and replayed
        _case("intersection_frames", "frames", "intersection", 21, 21, 30, 11, 11),
        # the three stages as separate calls (a program that looks at the poses and the table in between), odd
        # grid sizes, pedestrians that accelerate, a horizon that is no multiple of 32
        _case("stages_ragged", "stages", "accelerating", 19, 23, 37, 9, 13, weighted=True),
        # vehicles as convex outlines instead of rectangles
        _case("outlines_evaluate", "evaluate", "outlines", 21, 21, 30, 11, 11),
        # vehicles that follow lane paths under the lateral controller
        _case("lane_paths_evaluate", "evaluate", "lane_paths", 63, 7, 30, 11, 11),
        # the paper's own shape: an EGO of 6 x 343 hypotheses against ten objects of 6 x 7, 100 steps of 20 ms
        _case("ego_only_evaluate", "evaluate", "ego_only", 6, 343, 100, count=10),
        # requests that arrive together at the serving loop
        _case("serve_burst", "serve", "intersection", 21, 21, 30, 11, 11, count=48),
        # an ordinary batch of uneven scenes in one call, laid out anew on every call
        _case("batch24_call", "batch", "uneven", 0, 0, 0, count=24),
        # the large batch of uneven scenes, laid out once and replayed as a graph
        _case("batch256_plan", "plan", "uneven", 0, 0, 0, count=256),
        # 32 cars of 2048 hypotheses each: the largest single scene (1.0e11 pose tests, a 4.2 GB table)
        _case("cars32_evaluate", "evaluate", "cars", 64, 32, 50, count=32),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    scene = rng.choice(("crossing", "intersection", "intersection", "accelerating", "outlines", "lane_paths",
                        "ego_only", "uneven", "uneven", "cars", "cars"))
    weighted = rng.random() < 0.4
    if scene == "uneven":
        case = _case("", rng.choice(("batch", "plan")), scene, 0, 0, 0, count=_log_int(rng, 2, 160), sizes=rng.randint(1, 9999),
                     weighted=weighted)
    elif scene == "ego_only":
        case = _case("", rng.choice(("run", "evaluate")), scene, rng.randint(3, 12), _log_int(rng, 49, 343),
                     rng.randint(50, 120), count=rng.randint(2, 12), weighted=weighted)
    elif scene == "cars":
        case = _case("", "evaluate", scene, _log_int(rng, 8, 64), _log_int(rng, 5, 33), rng.randint(20, 50),
                     count=4 * rng.randint(2, 7), weighted=weighted)
    elif scene == "crossing":
        case = _case("", rng.choice(("run", "evaluate", "frames", "stages")), scene, rng.randint(3, 24),
                     rng.randint(1, 24), rng.randint(5, 60), weighted=weighted)
    else:
        call = rng.choice(("run", "evaluate", "frames", "stages", "serve"))
        n_str = 7 if scene == "lane_paths" else _log_int(rng, 5, 41)
        case = _case("", call, scene, _log_int(rng, 5, 41), n_str, rng.randint(15, 60), _log_int(rng, 3, 15),
                     _log_int(rng, 3, 15), count=rng.randint(8, 32) if call == "serve" else 1, weighted=weighted)
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------------------------
# what a program has in hand


def _scene(case, seed):
    """One scene of the case (``seed`` places its objects)."""
    na, nb, n = case["n_acc"], case["n_str"], case["n_steps"]
    kind = case["scene"]
    if kind == "crossing":
        sc = S.tiny_crossing(seed, start=18.0)
        objs = [dataclasses.replace(o, grid_a=S.accel_grid_paper(na, -6.0, 2.0), grid_b=S.linspace(-0.1, 0.1, nb))
                for o in sc.objects]
        return dataclasses.replace(sc, objects=objs, n_steps=n)
    if kind == "cars":
        return S.stress32(seed, case["count"], na, nb, n)
    if kind == "ego_only":
        sc = S.paper_s1s2(case["count"], na, seed)
        ego = dataclasses.replace(sc.objects[0], grid_b=S.linspace(-0.05, 0.05, nb))
        return dataclasses.replace(sc, objects=[ego] + sc.objects[1:], n_steps=n)
    sc = S.intersection11(seed, n, na, nb, case["n_ped_v"], case["n_ped_h"])
    if kind == "accelerating":
        return S.paper_pedestrians(sc, case["n_ped_v"], case["n_ped_h"], seed)
    if kind == "outlines":
        return S.with_outlines(sc, cut=0.35)
    if kind == "lane_paths":
        return S.with_lane_paths(sc)
    return sc


def _scenes(case, seed):
    """The scenes one pass evaluates."""
    if case["scene"] == "uneven":   # the batch's object and grid sizes are the case's, its initial states the seed's
        scenes = S.batch_scenarios(case["sizes"], case["count"])
        rng = np.random.default_rng(seed)
        for sc in scenes:
            for q, o in enumerate(sc.objects):
                ahead = rng.uniform(-1.0, 1.0)
                sc.objects[q] = dataclasses.replace(
                    o, x0=o.x0 + ahead * math.cos(o.psi0), y0=o.y0 + ahead * math.sin(o.psi0),
                    v0=rng.uniform(8.0, 15.0) if o.kind == S.VEHICLE else o.v0)
        return scenes
    if case["call"] == "serve":
        return [_scene(case, 1000 * seed + q) for q in range(case["count"])]
    return [_scene(case, seed)]


def _weights(case, scenes, seed):
    """The caller's weights per object of every scene (None: the library's uniform ones)."""
    if not case["weighted"]:
        return None
    rng = np.random.default_rng(seed)
    return [rng.uniform(0.05, 1.0, o.n_hyp).astype(np.float32) for sc in scenes for o in sc.objects]


def prepare(case, seed):
    scenes = _scenes(case, seed)
    weights = _weights(case, scenes, seed)
    call = case["call"]
    st = {"call": call}
    if call in ("batch", "plan", "frames"):
        st["batch"] = mhc.CBatch(scenes)
        info, _ = mhc.batch_layout(st["batch"])
        st["buffers"] = mhc.alloc_batch(info)
        st["weights"] = mhc.CWeights(weights)
        st["ctx"] = mhc.Context(0, max(8 << 20, info["scratch"] if call == "batch" else 0))
        if call != "batch":
            st["plan"] = mhc.Plan(st["ctx"], st["batch"], weights=st["weights"], buffers=st["buffers"])
        return st
    if call == "serve":
        st["requests"] = [mhc.as_c(sc) for sc in scenes]
        n = [sc.n_objects for sc in scenes]
        st["weights"] = [mhc.CWeights(None if weights is None else weights[sum(n[:q]): sum(n[:q + 1])])
                         for q in range(len(scenes))]
        # the outputs of all requests: request q's are row q
        st["out"] = {k: torch.zeros((len(scenes),) + shape, dtype=dt)
                     for k, (shape, dt) in mhc.risk_shapes(st["requests"][0]).items()}
        st["rows"] = [{k: v[q] for k, v in st["out"].items()} for q in range(len(scenes))]
        st["ctx"] = mhc.Context(0, 64 << 20)
        need = mhc.layout(st["requests"][0])["run_bytes"]
        st["server"] = mhc.Server(st["ctx"], 2 * len(scenes) * need)
        return st
    sc = st["scene"] = mhc.as_c(scenes[0])
    st["weights"] = mhc.CWeights(weights)
    lay = mhc.layout(sc)
    st["ctx"] = mhc.Context(0, max(8 << 20, lay["run_bytes"] if call == "run" else lay["scratch"]))
    if call == "run":
        st["out"] = mhc.alloc_risk(sc, device="cpu", pin=True)
        st["out_struct"] = mhc.risk_struct(st["out"])
    else:
        st["poses"] = mhc.alloc_poses(sc)
        st["table"] = torch.empty(lay["n_entries"], dtype=torch.int16, device="cuda")
        st["out"] = mhc.alloc_risk(sc)
    return st


# ---------------------------------------------------------------------------------------------------------
# one pass


def run(st):
    call, ctx = st["call"], st["ctx"]
    if call == "run":
        return {"risk": mhc.run(ctx, st["scene"], weights=st["weights"], out=st["out"], out_struct=st["out_struct"])}
    if call == "serve":
        server = st["server"]
        tickets = [server.submit(sc, w) for sc, w in zip(st["requests"], st["weights"])]
        for ticket, row in zip(tickets, st["rows"]):
            server.poll(ticket, row)
            server.release(ticket)
        return {"risk": st["out"]}
    if call == "evaluate":
        poses, table, out = mhc.evaluate(ctx, st["scene"], st["poses"], st["table"], st["weights"], st["out"])
    elif call == "stages":
        poses = mhc.generate(ctx, st["scene"], st["poses"])
        table = mhc.detect(ctx, st["scene"], poses, st["table"])
        out = mhc.assess(ctx, st["scene"], table, st["weights"], st["out"])
    elif call == "batch":
        poses, table, out = mhc.evaluate_batch(ctx, st["batch"], *st["buffers"][:2], weights=st["weights"],
                                               out=st["buffers"][2])
    else:
        if call == "frames":
            st["plan"].update(st["batch"])
        poses, table, out = st["plan"].launch()
    return {"poses": poses, "table": table, "risk": out}


def work(case):
    """Bytes: every pose and table entry the call returns written once (and read back once between separate calls),
    and the weights read.  Flops: the integration's sub-steps, and one distance test per trajectory pair (most of
    the others can be culled)."""
    scenes = _scenes(case, 1)
    poses = sum(o.n_hyp * sc.n_steps for sc in scenes for o in sc.objects)
    hyps = sum(o.n_hyp for sc in scenes for o in sc.objects)
    entries = sum(sc.n_traj_pairs() for sc in scenes)
    nbytes = 16.0 * poses + 2.0 * entries
    if case["call"] == "stages":
        nbytes *= 2
    if case["weighted"]:
        nbytes += 4.0 * hyps
    per_substep = 200.0 if case["scene"] == "lane_paths" else 115.0
    flops = sum(per_substep * o.n_hyp * sc.n_steps * sc.substeps for sc in scenes for o in sc.objects
                if o.kind == S.VEHICLE)
    return {"bytes": nbytes, "flops": flops + 5.0 * entries}


# ---------------------------------------------------------------------------------------------------------
# the floating outputs in 64 bits

_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _t64(v):
    return torch.as_tensor(np.asarray(v, np.float64), device=_DEV)


def _grid(o):
    """grid_a and grid_b values of every hypothesis of an object."""
    a, b = _t64(o.grid_a), _t64(o.grid_b)
    return a.repeat_interleave(b.numel()), b.repeat(a.numel())


def _cat(parts):
    return torch.cat(list(parts)) if parts else torch.zeros(0, dtype=torch.float64, device=_DEV)


def _vehicles(scenes, n_out, tau, substeps):
    """x, y, psi [n_out, hypotheses] of all vehicles: the one-track model with constant steering, or under the
    lateral controller where the object follows paths."""
    cars = [(sc, o) for sc in scenes for o in sc.objects if o.kind == S.VEHICLE]

    def each(f):
        return _cat([torch.full((o.n_hyp,), float(f(sc, o)), dtype=torch.float64, device=_DEV) for sc, o in cars])

    acc, delta = _cat([_grid(o)[0] for _, o in cars]), _cat([_grid(o)[1] for _, o in cars])
    prm = [S.DEFAULT_VEH_PARAMS if o.params is None else o.params for _, o in cars]
    m, iz, lf, lr, caf, car = (_cat([torch.full((o.n_hyp,), float(p[q]), dtype=torch.float64, device=_DEV)
                                     for (_, o), p in zip(cars, prm)]) for q in range(6))
    x, y, psi, v0 = (each(lambda sc, o, f=f: getattr(o, f)) for f in ("x0", "y0", "psi0", "v0"))
    kin = each(lambda sc, o: sc.model == S.MODEL_KIN) > 0
    follows = each(lambda sc, o: o.paths is not None) > 0
    path = torch.cat([_t64(o.paths).repeat(o.grid_a.size, 1, 1) if o.paths is not None else
                      torch.zeros((o.n_hyp, 3, 3), dtype=torch.float64, device=_DEV) for _, o in cars])
    delta = torch.where(follows, torch.zeros_like(delta), delta)
    ti, span = tau / substeps, lf + lr
    beta, r = torch.zeros_like(x), torch.zeros_like(x)
    ax, ay = acc.clone(), torch.zeros_like(x)
    stopped, any_path = torch.zeros_like(kin), bool(follows.any())
    out = torch.empty((3, n_out, x.numel()), dtype=torch.float64, device=_DEV)
    for n in range(n_out * substeps):
        v, v_next = v0 + n * (acc * ti), v0 + (n + 1) * (acc * ti)
        if any_path:
            t = n * ti
            sx, sy, spsi = path[:, 0 if t < 1.0 else (1 if t < 1.5 else 2)].unbind(1)
            px, py = x + 0.5 * v * torch.cos(psi + beta), y + 0.5 * v * torch.sin(psi + beta)
            d = (sy - py) * torch.cos(spsi) - (sx - px) * torch.sin(spsi)
            e = spsi - psi
            e = e - 2.0 * math.pi * torch.floor((e + math.pi) / (2.0 * math.pi))
            g = ((-0.018 * v + 1.5) * d).abs()
            cmd = ((g + 0.5) * d + (9.5 - g) * (3.8197 * e)) * math.pi / 180.0
            nxt = (delta + (cmd - delta).clamp(-0.5 * ti, 0.5 * ti)).clamp(-0.5, 0.5)
            delta = torch.where(follows & ~stopped, nxt, delta)
        low = kin | (v < 2.0)
        vs = v.clamp_min(1e-3)
        bd = -(caf + car) / (m * vs) * beta + ((car * lr - caf * lf) / (m * vs * vs) - 1.0) * r + caf / (m * vs) * delta
        rd = (car * lr - caf * lf) / iz * beta - (caf * lf * lf + car * lr * lr) / (iz * vs) * r + caf * lf / iz * delta
        tan_d = torch.tan(delta)
        b_low = torch.atan(lr * tan_d / span)
        b_use = torch.where(low, b_low, beta)
        r_use = torch.where(low, v * torch.cos(b_low) * tan_d / span, r)
        bd, rd = torch.where(low, 0.0, bd), torch.where(low, 0.0, rd)
        stop = (v_next < 0.0) & ~stopped
        go = ~stop & ~stopped
        cc, sc_ = torch.cos(psi + b_use), torch.sin(psi + b_use)
        cp, sp = torch.cos(psi), torch.sin(psi)
        d_stop = v * v / (2.0 * acc.abs().clamp_min(1e-30))
        half = ti * ti / 2.0
        x = x + torch.where(stop, cc * d_stop, torch.where(go, cc * v * ti + (cp * ax - sp * ay) * half, 0.0))
        y = y + torch.where(stop, sc_ * d_stop, torch.where(go, sc_ * v * ti + (sp * ax + cp * ay) * half, 0.0))
        psi = psi + torch.where(go, r_use * ti + rd * half, 0.0)
        cb, sb = torch.cos(b_use), torch.sin(b_use)
        w = v * (bd + r_use)
        ax, ay = torch.where(go, cb * acc - sb * w, ax), torch.where(go, sb * acc + cb * w, ay)
        beta, r = torch.where(go, b_use + bd * ti, beta), torch.where(go, r_use + rd * ti, r)
        stopped = stopped | stop
        if (n + 1) % substeps == 0:
            out[:, (n + 1) // substeps - 1] = torch.stack((x, y, psi))
    return out


def _pedestrian(o, n_out, tau):
    """x, y, psi [n_out, hypotheses]: constant heading and acceleration, the speed held at rest or at its cap."""
    a, b = _grid(o)
    accel = bool(o.flags & S.PED_ACCEL_GRID)
    v0, acc = (torch.full_like(a, o.v0), a) if accel else (a, torch.zeros_like(a))
    t = (torch.arange(n_out, dtype=torch.float64, device=_DEV) + 1.0)[:, None] * tau
    inf = torch.full_like(a, math.inf)
    one = torch.ones_like(a)
    speeds_up, brakes = (acc > 0) & (o.v_max > 0.0), acc < 0
    ts = torch.where(speeds_up, ((o.v_max - v0) / torch.where(speeds_up, acc, one)).clamp_min(0.0), inf)
    ts = torch.where(brakes, v0 / torch.where(brakes, -acc, one), ts)
    v_end = torch.where(brakes, 0.0, torch.where(v0 >= o.v_max, v0, torch.full_like(a, o.v_max)))
    before = torch.minimum(t, ts)
    after = torch.where(t > ts, (t - ts) * v_end, 0.0)
    s = v0 * before + 0.5 * acc * before * before + after
    psi = o.psi0 + b
    return torch.stack((o.x0 + torch.cos(psi) * s, o.y0 + torch.sin(psi) * s, psi.expand(n_out, -1)))


def _poses(scenes):
    """Per scene, per object: x, y, c, s [n_steps, hypotheses]."""
    tau, substeps = scenes[0].tau, scenes[0].substeps
    longest = max(sc.n_steps for sc in scenes)
    cars, at, out = _vehicles(scenes, longest, tau, substeps), 0, []
    for sc in scenes:
        mine = []
        for o in sc.objects:
            if o.kind == S.VEHICLE:
                x, y, psi = cars[:, : sc.n_steps, at: at + o.n_hyp]
                at += o.n_hyp
            else:
                x, y, psi = _pedestrian(o, sc.n_steps, tau)
            mine.append((x, y, torch.cos(psi), torch.sin(psi)))
        out.append(mine)
    return out


def _corners(o, pose):
    """World vertices [n, 2] of a vehicle, each [steps, hypotheses]."""
    body = o.outline if o.outline is not None else S.chamfered_outline(o.length, o.width, 0.0)
    body = np.asarray(body, np.float64)
    if np.sum(body[:, 0] * np.roll(body[:, 1], -1) - np.roll(body[:, 0], -1) * body[:, 1]) < 0:
        body = body[::-1]
    x, y, c, s = pose
    return [(x + c * p - s * q, y + s * p + c * q) for p, q in body]


def _separates(va, vb):
    """Whether an edge of outline a (rows) has all of outline b (columns) strictly outside: [steps, h_a, h_b]."""
    found = None
    for (px, py), (qx, qy) in zip(va, va[1:] + va[:1]):
        nx, ny = qy - py, px - qx                       # outward: the vertices run counter-clockwise
        h = nx * px + ny * py
        lo = None
        for wx, wy in vb:
            d = nx[:, :, None] * wx[:, None, :] + ny[:, :, None] * wy[:, None, :]
            lo = d if lo is None else torch.minimum(lo, d)
        sep = lo > h[:, :, None]
        found = sep if found is None else found | sep
    return found


def _near(va, cx, cy, radius):
    """Whether discs (columns) touch outlines (rows): [steps, h_a, h_b]."""
    inside, d2 = None, None
    for (px, py), (qx, qy) in zip(va, va[1:] + va[:1]):
        px, py, qx, qy = (w[:, :, None] for w in (px, py, qx, qy))
        ex, ey, ux, uy = qx - px, qy - py, cx[:, None, :] - px, cy[:, None, :] - py
        left = ex * uy - ey * ux >= 0.0
        t = ((ux * ex + uy * ey) / (ex * ex + ey * ey)).clamp(0.0, 1.0)
        d = (ux - t * ex) ** 2 + (uy - t * ey) ** 2
        inside = left if inside is None else inside & left
        d2 = d if d2 is None else torch.minimum(d2, d)
    return inside | (d2 <= radius * radius)


def _first_steps(sc, poses, a, b):
    """[h_a, h_b] first overlapping step of objects a and b (-1: none)."""
    oa, ob = sc.objects[a], sc.objects[b]
    rows = max(1, int(4e7 / (sc.n_steps * ob.n_hyp)))
    out = []
    vb = _corners(ob, poses[b]) if ob.kind == S.VEHICLE else None
    for i in range(0, oa.n_hyp, rows):
        pa = [w[:, i: i + rows] for w in poses[a]]
        va = _corners(oa, pa) if oa.kind == S.VEHICLE else None
        if va is not None and vb is not None:
            hit = ~(_separates(va, vb) | _separates(vb, va).transpose(1, 2))
        elif va is not None:
            hit = _near(va, poses[b][0], poses[b][1], ob.radius)
        elif vb is not None:
            hit = _near(vb, pa[0], pa[1], oa.radius).transpose(1, 2)
        else:
            dx, dy = poses[b][0][:, None, :] - pa[0][:, :, None], poses[b][1][:, None, :] - pa[1][:, :, None]
            hit = dx * dx + dy * dy <= (oa.radius + ob.radius) ** 2
        out.append(torch.where(hit.any(0), hit.to(torch.int8).argmax(0), -1))
    return torch.cat(out)


def _risk(sc, poses, weights):
    """The floating risk outputs of one scene (None in the place of the integer ones)."""
    n, ego = sc.n_steps, sc.ego
    p = [_t64(w if w is not None else np.ones(o.n_hyp)) for o, w in zip(sc.objects, weights)]
    p = [w / w.sum() for w in p]
    he, no = sc.objects[ego].n_hyp, sc.n_objects
    mass = torch.zeros((he, no), dtype=torch.float64, device=_DEV)
    lsum = torch.zeros((he, n, no), dtype=torch.float64, device=_DEV)
    total, by_step = [], []
    for a, b in sc.pairs():
        first = _first_steps(sc, poses, a, b)
        w = p[a][:, None] * p[b][None, :]
        hist = torch.zeros(n + 1, dtype=torch.float64, device=_DEV).index_add_(0, (first + 1).reshape(-1), w.reshape(-1))
        by_step.append(hist[1:])
        total.append(hist[1:].sum())
        if ego in (a, b):
            co, f = (b, first) if a == ego else (a, first.T)
            hit = f >= 0
            mass[:, co] = torch.where(hit, p[co][None, :], 0.0).sum(1)
            terms = torch.where(hit, -torch.log1p(-p[co].clamp_max(1.0 - 1e-16))[None, :], 0.0)
            lsum[:, :, co] = torch.zeros((he, n + 1), dtype=torch.float64, device=_DEV).scatter_add_(1, f + 1, terms)[:, 1:]
    cells = lsum.reshape(he, -1)
    before = torch.cumsum(cells, 1) - cells
    gain = (torch.exp(-before) * -torch.expm1(-cells)).reshape(he, n, no)
    share = p[ego][:, None, None] * gain
    naive, cond, indep = mass.sum(1), gain.sum((1, 2)), 1.0 - torch.prod(1.0 - mass, 1)
    scalars = torch.stack([(p[ego] * v).sum() for v in (naive, cond, indep)] + [torch.zeros_like(naive[0])])
    return dict(count=None, count_k=None, P=torch.stack(total), H=torch.stack(by_step), naive=naive, cond=cond,
                indep=indep, hits=None, attr_obj=share.sum((0, 1)), attr_step=share.sum((0, 2)), scalars=scalars,
                escape=None, n_escape=None)


def exact(case, seed):
    scenes = _scenes(case, seed)
    weights = _weights(case, scenes, seed)
    poses = _poses(scenes)
    risk = None
    if sum(sc.n_tests() for sc in scenes) <= (5e9 if case["scene"] == "outlines" else 2e10):   # some 10 seconds
        at, parts = 0, []
        for sc, ps in zip(scenes, poses):
            parts.append(_risk(sc, ps, [None] * sc.n_objects if weights is None else weights[at: at + sc.n_objects]))
            at += sc.n_objects
        if case["call"] == "serve":
            risk = {k: None if v is None else torch.stack([q[k] for q in parts]) for k, v in parts[0].items()}
        elif case["call"] in ("batch", "plan", "frames"):
            risk = {k: None if v is None else torch.cat([q[k].reshape(-1) for q in parts]) for k, v in parts[0].items()}
        else:
            risk = parts[0]
    if case["call"] in ("run", "serve"):
        return None if risk is None else {"risk": risk}
    planes = {k: torch.cat([o[q].reshape(-1) for ps in poses for o in ps]) for q, k in enumerate(("x", "y", "c", "s"))}
    return {"poses": planes, "table": None, "risk": risk}

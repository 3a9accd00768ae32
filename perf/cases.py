"""Cases of the batched IK path, measured through the package's public entry points.

A user of this library registers a robot (and a scene) once, then solves poses: one at a
time in a control loop, a hundred in an evaluation set, a million candidates in a planner's
or data generator's batch.  The cases are those calls, with the sizes of the repository's
own workloads (``inputs.py``) and of the paper's tables, plus two of the stages that a program
calls on its own: forward kinematics and the collision filter.

Targets are poses of collision-free joint samples.  Their kinematics and the collision tests
behind the sampling are written here in plain torch, so the inputs depend on the seed alone.
"""
import math

import numpy as np
import torch

from paper_2510_07514_gb300 import api, hjcd, inputs

# ------------------------------------------------------------------ robots

_ROBOTS = {}


def _robot(name):
    """The description of a robot: "panda", "panda60" (with 60 link spheres), "chainN" (N joints
    of chained Panda copies), "randomK" (row K of the eight random chains, with link spheres)."""
    if name not in _ROBOTS:
        if name == "panda":
            r = inputs.panda()
        elif name == "panda60":
            r = inputs.panda_with_spheres(np.random.default_rng(inputs.CFG_SEED[2]))
        elif name.startswith("chain"):
            r = inputs.dof_scaling_robot(int(name[5:]))
        else:
            for k, c in enumerate(inputs.cfg3_chains()):
                _ROBOTS["random%d" % k] = c
            r = _ROBOTS[name]
        _ROBOTS[name] = r
    return _ROBOTS[name]


# A program keeps one context for its life, with its robots registered once.
_CTX = {}


def _context():
    if "solve" not in _CTX:
        _CTX["solve"] = (api.Context(0), {})
    return _CTX["solve"][0]


def _robot_id(name):
    ctx, ids = _context(), _CTX["solve"][1]
    if name not in ids:
        ids[name] = ctx.add_robot(_robot(name))
    return ids[name]


def _server():
    """The serving program's context: its robots registered, its loop running."""
    if "serve" not in _CTX:
        ctx = api.Context(0)
        ids = {k: ctx.add_robot(_robot("random%d" % k)) for k in inputs.CFG4_ROBOTS}
        hjcd.hjcd_server_start(ctx.h, max_inflight=3)
        _CTX["serve"] = (ctx, ids)
    return _CTX["serve"]


# ------------------------------------------- plain kinematics and collision

def _frames(rob, theta):
    """Body frames 0..n+1 of joint vectors theta [P, n] (64 bits): rotations [P, n+2, 3, 3], origins [P, n+2, 3]."""
    P, dev = theta.shape[0], theta.device
    f64 = dict(dtype=torch.float64, device=dev)
    T = torch.eye(4, **f64).expand(P, 4, 4)
    out = [T]
    # the device holds its tables in 32 bits
    a, al, d, off = (np.asarray(v, np.float32).astype(np.float64) for v in (rob.a, rob.alpha, rob.d, rob.theta_off))
    for j in range(rob.n):
        th = theta[:, j] + off[j]
        c, s = torch.cos(th), torch.sin(th)
        ca, sa = math.cos(al[j]), math.sin(al[j])
        z, o = torch.zeros_like(c), torch.ones_like(c)
        A = torch.stack([c, -s, z, a[j] * o,
                         s * ca, c * ca, -sa * o, -d[j] * sa * o,
                         s * sa, c * sa, ca * o, d[j] * ca * o,
                         z, z, z, o], 1).reshape(P, 4, 4)
        T = T @ A
        out.append(T)
    out.append(T @ torch.tensor(np.asarray(rob.flange, np.float32).astype(np.float64), **f64))
    M = torch.stack(out, 1)
    return M[:, :, :3, :3], M[:, :, :3, 3]


def _pose(R, p):
    """Poses px py pz qw qx qy qz (w >= 0) of rotations R [P, 3, 3] and positions p."""
    m = lambda i, j: R[:, i, j]  # noqa: E731
    tr = m(0, 0) + m(1, 1) + m(2, 2)
    q4 = torch.stack([1 + tr, 1 + 2 * m(0, 0) - tr, 1 + 2 * m(1, 1) - tr, 1 + 2 * m(2, 2) - tr], 1)  # 4 x^2 of each part
    a, b, c = m(2, 1) - m(1, 2), m(0, 2) - m(2, 0), m(1, 0) - m(0, 1)
    d, e, f = m(0, 1) + m(1, 0), m(0, 2) + m(2, 0), m(1, 2) + m(2, 1)
    rows = torch.stack([torch.stack([q4[:, 0], a, b, c], 1), torch.stack([a, q4[:, 1], d, e], 1),
                        torch.stack([b, d, q4[:, 2], f], 1), torch.stack([c, e, f, q4[:, 3]], 1)], 1)
    k = q4.argmax(1)
    q = rows[torch.arange(len(k), device=R.device), k]
    q = q / q.norm(dim=1, keepdim=True)
    return torch.cat([p, torch.where(q[:, :1] < 0, -q, q)], 1)


def _link_spheres(rob, R, p):
    """World centres [P, n_sph, 3] and radii [n_sph] of the link spheres."""
    b = torch.as_tensor(np.asarray(rob.sph_body, np.int64), device=p.device)
    s = torch.as_tensor(np.asarray(rob.sph_xyzr, np.float64), device=p.device)
    return (R[:, b] @ s[:, :3, None]).squeeze(-1) + p[:, b], s[:, 3]


def _free(rob, scene, theta):
    """Which joint vectors touch neither themselves nor the scene."""
    R, p = _frames(rob, theta)
    if not len(rob.sph_body):
        return torch.ones(len(theta), dtype=torch.bool, device=theta.device)
    c, r = _link_spheres(rob, R, p)
    body = np.asarray(rob.sph_body)
    ign = np.asarray(rob.ignore) != 0
    i, j = np.nonzero(np.triu(~(ign | ign.T)[body[:, None], body[None, :]], 1))
    i, j = (torch.as_tensor(v, device=theta.device) for v in (i, j))
    hit = torch.zeros(len(theta), dtype=torch.bool, device=theta.device)
    hit |= ((c[:, i] - c[:, j]).square().sum(-1) < (r[i] + r[j]).square()).any(1)
    if scene is not None and len(scene.sph_xyzr):
        o = torch.as_tensor(scene.sph_xyzr, device=theta.device)
        d2 = (c[:, :, None] - o[None, None, :, :3]).square().sum(-1)
        hit |= (d2 < (r[:, None] + o[None, :, 3]).square()).flatten(1).any(1)
    if scene is not None and len(scene.box_lohi):
        o = torch.as_tensor(scene.box_lohi, device=theta.device)
        x = c[:, :, None]
        d2 = (x - torch.minimum(torch.maximum(x, o[:, :3]), o[:, 3:])).square().sum(-1)
        hit |= (d2 < r[:, None].square()).flatten(1).any(1)
    return ~hit


def _samples(rng, rob, count, scene=None, checked=True):
    """count joint vectors uniform in the limits (64 bits, on the GPU), collision-free ones when checked."""
    draw = lambda k: torch.as_tensor(inputs.joint_samples(rng, rob, k), device="cuda")  # noqa: E731
    if not checked:
        return draw(count)
    got, have = [], 0
    for _ in range(64):
        th = draw(min(4096, max(64, 4 * (count - have))))
        th = th[_free(rob, scene, th)]
        got.append(th)
        have += len(th)
        if have >= count:
            break
    else:
        got.append(draw(count - have))  # a scene with hardly any room: such targets have no witness
    return torch.cat(got)[:count]


def _roomy_scene(rng, rob, count, n_sph, n_box):
    """A scene and collision-free joint samples in it: one with half the obstacles where there is no room."""
    for _ in range(8):
        scene = inputs.random_scene(rng, n_sph, n_box)
        if bool(_free(rob, scene, _samples(rng, rob, 256, checked=False)).any()):
            break
        n_sph, n_box = n_sph // 2, n_box // 2
    return scene, _samples(rng, rob, count, scene)


def _targets(rob, theta):
    R, p = _frames(rob, theta)
    return _pose(R[:, -1], p[:, -1]).float()


def _grid_scene(rng, rob, theta, n_obstacles):
    """Small obstacle spheres on a jittered lattice, those that touch one of the configurations left out."""
    nodes = inputs.jittered_grid_nodes(rng)
    node = torch.as_tensor(nodes, dtype=torch.float32, device="cuda")
    R, p = _frames(rob, theta)
    c, r = _link_spheres(rob, R, p)
    c, r = c.reshape(-1, 3).float(), r.float().repeat(len(theta))
    touched = torch.zeros(len(nodes), dtype=torch.bool, device="cuda")
    for k in range(0, len(c), 2048):
        d2 = sum((c[k:k + 2048, None, a] - node[None, :, a]).square() for a in range(3))
        touched |= (d2 < (r[k:k + 2048, None] + node[None, :, 3]).square()).any(0)
    keep = nodes[~touched.cpu().numpy()][:n_obstacles]
    return inputs.Scene(keep, np.zeros((0, 6)))


# ------------------------------------------------------------------- cases

def listed():
    return [
        # one pose for a teleoperated arm, few seeds: the smallest call, pure latency
        dict(name="pose_1x64", kind="solve", robot="panda", targets=1, seeds=64, top_k=1, spheres=0, boxes=0, host=False),
        # the paper's batch of 1000 seeds on one pose, as a program with host data calls it
        dict(name="pose_1x1000", kind="solve", robot="panda60", targets=1, seeds=1000, top_k=1, spheres=0, boxes=0, host=True),
        # a tracking frame: moving obstacles rewritten, one pose, the solution nearest to the arm
        dict(name="track_1x1000", kind="track", robot="panda60", targets=1, seeds=1000, top_k=1, spheres=24, boxes=0, host=False),
        # the paper's longest chain and largest batch, several solutions kept
        dict(name="chain24_1x2000", kind="solve", robot="chain24", targets=1, seeds=2000, top_k=16, spheres=0, boxes=0, host=False),
        # a fixed small batch captured once and replayed by a control loop
        dict(name="graph_16x64", kind="graph", robot="panda", targets=16, seeds=64, top_k=4, spheres=0, boxes=0, host=False),
        # an evaluation set of about a hundred poses in a cluttered scene, from host data
        dict(name="poses_97x1000", kind="solve", robot="panda60", targets=97, seeds=1000, top_k=1, spheres=200, boxes=20, host=True),
        # the benchmark's step: a thousand poses, a million candidates
        dict(name="poses_1000x1000", kind="solve", robot="panda60", targets=1000, seeds=1000, top_k=1, spheres=200, boxes=20, host=False),
        # eight chains of 6 to 20 joints with uneven seed counts, packed into one call
        dict(name="uneven_8x40", kind="batch", robot="random", targets=40, seeds=4096, top_k=1, spheres=100, boxes=0, host=False),
        # many seeds in a scene of thousands of small obstacles, sixteen solutions each (a planner's goal sets)
        dict(name="grid_2000x4096", kind="solve", robot="panda60", targets=2000, seeds=4096, top_k=16, spheres=5000, boxes=0, host=False),
        # a burst of requests of different robots, scenes and sizes through the serving loop
        dict(name="serve_20", kind="serve", robot="random", targets=8, seeds=4096, top_k=1, spheres=500, boxes=0, host=True, requests=20),
        # the collision filter on its own: every configuration of a planner's sample set
        dict(name="collide_400k", kind="collide", robot="panda60", targets=400000, seeds=1, top_k=1, spheres=200, boxes=20, host=False),
        # forward kinematics on its own: poses of a data generator's joint samples
        dict(name="fk_1M", kind="fk", robot="panda", targets=1000000, seeds=1, top_k=1, spheres=0, boxes=0, host=False),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "track", "graph", "batch", "serve", "collide", "fk"])
    c = dict(kind=kind, robot="random", top_k=1, targets=1, seeds=1, spheres=0, boxes=0, host=False)
    if kind == "serve":
        c.update(targets=rng.randint(1, 8), seeds=_log_int(rng, 64, 4096), spheres=rng.randint(0, 500), host=True,
                 requests=rng.randint(2, 20))
        return c
    if kind == "batch":
        c.update(targets=_log_int(rng, 1, 100), seeds=_log_int(rng, 64, 4096), spheres=rng.randint(0, 100),
                 top_k=rng.choice([1, 4, 16]), host=rng.random() < 0.3)
        return c
    if kind in ("collide", "fk"):
        c.update(targets=_log_int(rng, 100, 400000 if kind == "collide" else 2000000))
        c.update(robot=rng.choice(["panda60", "random%d" % rng.randrange(8)]))
        if kind == "collide":
            c.update(spheres=rng.randint(0, 400), boxes=rng.randint(0, 20))
        return c
    c["robot"] = rng.choice(["panda", "panda60", "panda60", "chain12", "chain18", "chain24", "random%d" % rng.randrange(8)])
    scene = c["robot"] == "panda60" or c["robot"].startswith("random")
    c.update(top_k=rng.choice([1, 4, 16]), seeds=_log_int(rng, 10, 4096))
    if kind == "track":
        c.update(spheres=rng.randint(1, 48) if scene else 0)
    elif kind == "graph":
        c.update(targets=_log_int(rng, 1, 200), spheres=rng.randint(0, 100) if scene else 0)
    else:
        c.update(targets=_log_int(rng, 1, 2000), host=rng.random() < 0.4)
        if scene:
            c.update(spheres=rng.choice([0, rng.randint(10, 250), 5000]) if c["robot"] == "panda60" else rng.randint(0, 100))
            c.update(boxes=rng.randint(0, 20) if 0 < c["spheres"] < 5000 else 0)
    # no more than the largest listed case's work
    c["targets"] = max(1, min(c["targets"], int(4e6 / (c["seeds"] * _robot(c["robot"]).n / 7))))
    return c


class _State:
    def __init__(self, **kw):
        self.__dict__.update(kw)
        self.ctx = _context()

    def __del__(self):
        if getattr(self, "graph", None) is not None:
            hjcd.hjcd_graph_destroy(self.graph)


def _serve_state(case, rng):
    """Requests of the serving program: each one of its robots, a scene of its own, one to `targets` poses."""
    ctx, ids = _server()
    items, outs = [], []
    for r in range(case["requests"]):
        k = inputs.CFG4_ROBOTS[(3 * r) % 4]
        rob = _robot("random%d" % k)
        sc, th = _roomy_scene(rng, rob, 1 + (5 * r) % case["targets"], int(rng.integers(0, case["spheres"] + 1)), 0)
        tg = _targets(rob, th).cpu()
        seeds = int(inputs.log_uniform_counts(rng, 1, 32, case["seeds"])[0])
        it, out = ctx.batch_item(ids[k], -1, tg, seeds, case["top_k"], int(rng.integers(0, 2 ** 63 - 1)), rob.n,
                                 spheres=np.asarray(sc.sph_xyzr, np.float32))
        items.append(it)
        outs.append(out)
    keep, ctx._keep = ctx._keep, []  # the request's arrays live with the state
    return _State(kind="serve", server=ctx, items=items, outs=outs, keep=keep)


def prepare(case, seed):
    rng = np.random.default_rng(int(seed))
    kind, host = case["kind"], case["host"]
    dev = "cpu" if host else "cuda"
    if kind == "serve":
        return _serve_state(case, rng)
    ctx = _context()
    if kind == "batch":
        scene = inputs.random_scene(rng, case["spheres"], case["boxes"])
        sid = ctx.set_scene(scene)
        items, outs = [], []
        for k in range(8):
            rob = _robot("random%d" % k)
            tg = _targets(rob, _samples(rng, rob, case["targets"], scene)).to(dev)
            spt = inputs.log_uniform_counts(rng, case["targets"], 32, case["seeds"]).astype(np.int32)
            it, out = ctx.batch_item(_robot_id("random%d" % k), sid, tg, int(spt.max()), case["top_k"],
                                     int(rng.integers(0, 2 ** 63 - 1)), rob.n, samples_per_target=spt)
            items.append(it)
            outs.append(out)
        keep, ctx._keep = ctx._keep, []
        return _State(kind=kind, items=items, outs=outs, keep=keep)

    rob, rid = _robot(case["robot"]), _robot_id(case["robot"])
    if kind in ("collide", "fk"):
        th = _samples(rng, rob, case["targets"], checked=False).float().t().contiguous()
        sid = ctx.set_scene(inputs.random_scene(rng, case["spheres"], case["boxes"])) if kind == "collide" and case["spheres"] + case["boxes"] else -1
        return _State(kind=kind, rid=rid, sid=sid, theta=th)

    scene, sid = None, -1
    if case["spheres"] >= 1000:
        th = _samples(rng, rob, case["targets"])
        scene = _grid_scene(rng, rob, th, case["spheres"])
    elif case["spheres"] + case["boxes"]:
        scene, th = _roomy_scene(rng, rob, case["targets"], case["spheres"], case["boxes"])
    else:
        th = _samples(rng, rob, case["targets"])
    if scene is not None:
        sid = ctx.set_scene(scene)
    s = _State(kind=kind, rid=rid, sid=sid, scene=scene, n=rob.n, targets=_targets(rob, th).to(dev), seeds=case["seeds"],
               top_k=case["top_k"], seed=int(rng.integers(0, 2 ** 63 - 1)))
    if kind == "track":
        s.q_current = torch.as_tensor(inputs.joint_samples(rng, rob, case["targets"]), dtype=torch.float32).to(dev)
    if kind == "graph":
        s.item, s.out = ctx.batch_item(rid, sid, s.targets, s.seeds, s.top_k, s.seed, s.n)
        s.keep, ctx._keep = ctx._keep, []
        torch.cuda.synchronize()
        s.graph = hjcd.hjcd_graph_create(ctx.h, [s.item])
    return s


def run(s):
    ctx = s.ctx
    if s.kind == "fk":
        return ctx.fk(s.rid, s.theta)
    if s.kind == "collide":
        return ctx.collide(s.rid, s.sid, s.theta)
    if s.kind == "batch":
        ctx.solve_batch(s.items)
        return s.outs
    if s.kind == "graph":
        hjcd.hjcd_graph_launch(ctx.h, s.graph)
        return s.out
    if s.kind == "serve":
        ids = [hjcd.hjcd_submit(s.server.h, it) for it in s.items]
        for i in ids:
            info = hjcd.hjcd_wait(s.server.h, i)
            if info.status:
                raise RuntimeError("request failed: %d" % info.status)
        return s.outs
    if s.kind == "track":
        if s.scene is not None:
            ctx.set_scene(s.scene, s.sid)  # the frame's obstacles
        return ctx.solve(s.rid, s.sid, s.targets, s.seeds, s.top_k, s.seed, s.n, q_current=s.q_current)
    return ctx.solve(s.rid, s.sid, s.targets, s.seeds, s.top_k, s.seed, s.n)


# Iterations a candidate takes on average (counted by the library on the Panda batch) and the
# operations of one, with n joints: 29 of at most 32 PO-CCD iterations, 7.2 PJ-IK iterations with
# two further kinematics passes each; a collision check takes about 700 sphere tests.
def _solve_flops(candidates, n):
    return candidates * (29 * (252 * n + 301) + 7.2 * (173 * n + 410 + 2 * (56 * n + 166)))


def _mean_log_uniform(lo, hi):
    return (hi - lo) / math.log(hi / lo)


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        robots = range(8) if kind == "batch" else inputs.CFG4_ROBOTS
        n = sum(_robot("random%d" % k).n for k in robots) / len(robots)
        targets = 8 * case["targets"] if kind == "batch" else case["requests"] * (case["targets"] + 1) / 2
        seeds = _mean_log_uniform(32, max(case["seeds"], 33))
    else:
        n, targets, seeds = _robot(case["robot"]).n, case["targets"], case["seeds"]
    if kind == "fk":
        return dict(bytes=4 * targets * (n + 7), flops=targets * (56 * n + 60))
    if kind == "collide":
        ns = len(_robot(case["robot"]).sph_body)
        tests = 700 if case["spheres"] + case["boxes"] else 200
        return dict(bytes=targets * (4 * n + 1) + 16 * (ns + case["spheres"] + 2 * case["boxes"]),
                    flops=targets * (18 * ns + 54 * n + 63 + 10 * tests))
    return dict(bytes=targets * (28 + 4 + 4 * case["top_k"] * (n + 2)) + 16 * (case["spheres"] + 2 * case["boxes"]),
                flops=_solve_flops(targets * seeds, n))


def exact(case, seed):
    """Forward kinematics in 64 bits.  The solves are randomised searches whose result has no
    closed form (each rounding may change a decision), and the filter's verdicts are whole numbers."""
    if case["kind"] != "fk":
        return None
    rob = _robot(case["robot"])
    s = prepare(case, seed)
    out = []
    for th in s.theta.t().double().split(65536):
        R, p = _frames(rob, th)
        out.append(_pose(R[:, -1], p[:, -1]))
    return torch.cat(out)

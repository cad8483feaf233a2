"""The performance cases of this framework: what its users have it do, over the range of sizes.

Most cases are a rollout as a controller, a planner or a learning loop makes it: the state
goes in from pinned host memory, the simulation takes its time steps, and the whole state
(poses and velocities of every body, positions and velocities of every node) comes back.
The state is written before every pass, so that a pass does the same work however often it
is repeated.  Iteration counts are fixed per step, as the paper runs its scenes and as a
real-time loop budgets them, except in FP64 cases that stop at the tolerance.  The two
last cases are the learned warm start's network: inference over the interfaces of a batch
of scenes, and the gradients of one training minibatch.

The mixed form (FP32 iterations) returns its state in FP32, the precision it works in; the
FP64 form returns FP64.
"""
import math

import numpy as np
import torch

import scenegen as sg
from paper_2302_14344_gb300 import subadmm as sa
from paper_2302_14344_gb300 import warmstart as ws

NET = [32, 256, 256, 256, 7]          # the warm-start network's widths


def listed():
    return [
        # one small mechanism stepped in a control loop: 8 links, one step per call, all
        # latency (the smallest call there is)
        dict(name="chain8_fp64", kind="chain", links=8, per_sub=2, mixed=False, iters=100,
             steps=1),
        # a learning loop's environments: 64 legged robots at touchdown, the iterations that
        # the contact phase needs on average, two steps of 2 ms per action
        dict(name="robots64_mixed", kind="robots", robots=64, mixed=True, iters=600, steps=2),
        # the same robots in reference precision, every step run to r_p <= 1e-6
        dict(name="robots48_fp64_tol", kind="robots", robots=48, mixed=False, iters=1000,
             tol=1e-6, steps=6),
        # a batch of unlike scenes (chains and elastic blocks of 6 to 240 DOF) solved side by
        # side, the iterations that the tolerance takes on average
        dict(name="batched384_mixed", kind="batched", scenes=384, mixed=True, iters=300,
             steps=1),
        # a smaller batch in reference precision
        dict(name="batched64_fp64", kind="batched", scenes=64, mixed=False, iters=100, steps=1),
        # the large elastic beam (20,000 nodes, 64 slabs, gripper): factors kept over the run,
        # the iterations that the tolerance takes on average, three steps per call
        dict(name="beam64_mixed", kind="beam", slabs=64, ny=10, nz=10, corot=False, mixed=True,
             iters=550, steps=3),
        # the same beam co-rotational, as in the paper: every step rebuilds and refactorises
        # all slabs, 90 iterations
        dict(name="beam64_corot_mixed", kind="beam", slabs=64, ny=10, nz=10, corot=True,
             mixed=True, iters=90, steps=1),
        # a shorter co-rotational beam in reference precision
        dict(name="beam16_corot_fp64", kind="beam", slabs=16, ny=10, nz=10, corot=True,
             mixed=False, iters=60, steps=1),
        # the paper's cable scene at its 90 iterations: one scene of many small subsystems
        dict(name="cable640_mixed", kind="cable", segments=640, mixed=True, iters=90, steps=2),
        # the paper's granular scene at its 30 iterations: contact-heavy, one body a subsystem
        dict(name="stir216_mixed", kind="stir", side=6, layers=6, pj=False, mixed=True,
             iters=30, steps=1),
        # the warm-start network over the interfaces of some thousand scenes
        dict(name="net_infer", kind="net_infer", batch=131071),
        # the network's gradients for one training minibatch
        dict(name="net_gradients", kind="net_grad", batch=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "robots", "batched", "beam", "beam", "cable", "stir", "stir",
                       "generic", "net_infer", "net_grad"])
    mixed = rng.random() < 0.5
    if kind == "chain":
        per = rng.choice([1, 2, 4])
        return dict(kind=kind, links=per * _log(rng, 2, 16), per_sub=per, mixed=mixed,
                    iters=_log(rng, 30, 300), steps=rng.randint(1, 4))
    if kind == "robots":
        c = dict(kind=kind, robots=_log(rng, 1, 128), mixed=mixed, iters=_log(rng, 30, 600),
                 steps=rng.randint(1, 3))
        if not mixed and rng.random() < 0.5:
            c.update(iters=1000, tol=1e-6, steps=rng.randint(3, 6))
        return c
    if kind == "batched":
        n = _log(rng, 4, 384 if mixed else 96)
        return dict(kind=kind, scenes=n, mixed=mixed,
                    iters=_log(rng, 30, 300 if mixed else 100), steps=1)
    if kind == "beam":
        corot = rng.random() < 0.5
        slabs = _log(rng, 2, 16 if corot and not mixed else 64)
        return dict(kind=kind, slabs=slabs, ny=rng.randint(4, 10), nz=rng.randint(4, 10),
                    corot=corot, mixed=mixed, iters=_log(rng, 30, 90 if corot else 300),
                    steps=1)
    if kind == "cable":
        return dict(kind=kind, segments=4 * _log(rng, 6, 160), mixed=mixed,
                    iters=_log(rng, 30, 90), steps=rng.randint(1, 2))
    if kind == "stir":
        return dict(kind=kind, side=rng.randint(3, 6), layers=rng.randint(2, 6),
                    pj=rng.random() < 0.3, mixed=mixed, iters=_log(rng, 30, 90),
                    steps=1)
    if kind == "generic":
        return dict(kind=kind, scenes=_log(rng, 1, 16), subs=rng.randint(2, 12),
                    dof=_log(rng, 4, 96), extra=rng.randint(0, 12), mixed=mixed,
                    iters=_log(rng, 30, 200), steps=1)
    if kind == "net_infer":
        return dict(kind=kind, batch=_log(rng, 1, 600000))
    return dict(kind=kind, batch=_log(rng, 64, 8192))


# ---------------------------------------------------------------------------- the inputs

def _ground(scene, rng):
    """Lowers a scene until its lowest contact point touches the plane, falling at up to
    0.3 m/s (a scene that has just landed)."""
    low = math.inf
    for f in scene.ifs:
        if f.kind != sg.PLANE_CONTACT:
            continue
        s, k = f.a
        if hasattr(scene.subs[s], "bodies"):
            b = scene.subs[s].bodies[k]
            low = min(low, b.p[2] + (_rot(b.q[None])[0] @ f.anchor_a)[2])
        else:
            low = min(low, scene.subs[s].x[3 * k + 2])
    d, v = (0.0 if low == math.inf else -low), -float(rng.uniform(0.0, 0.3))
    for s in scene.subs:
        if hasattr(s, "bodies"):
            for b in s.bodies:
                b.p = b.p + np.array([0.0, 0.0, d])
                b.v = b.v + np.array([0.0, 0.0, v])
        else:
            s.x = s.x.copy()
            s.X0 = s.X0.copy()
            s.v = s.v.copy()
            s.x[2::3] += d
            s.X0[2::3] += d
            s.v[2::3] += v


def _problem(case, seed):
    kind, it = case["kind"], dict(max_iters=case["iters"], tol_primal=case.get("tol", -1.0))
    rng = np.random.default_rng([seed, 17])
    if kind == "chain":
        return sg.chain(seed, n_links=case["links"], links_per_sub=case["per_sub"], **it)
    if kind == "robots":
        p = sg.robots(seed, n_robots=case["robots"], drop=(0.0, 1e-3), **it)
        for s in p.scenes:
            _ground(s, rng)
        return p
    if kind == "batched":
        # (the batch's make-up goes with its size, its state with the seed)
        p = sg.batched(case["scenes"], n_scenes=case["scenes"], **it)
        for s in p.scenes:
            _ground(s, rng)
            for u in s.subs:
                v = rng.uniform(-0.1, 0.1, 3)
                if hasattr(u, "bodies"):
                    for b in u.bodies:
                        b.v = b.v + v
                        b.w = b.w + rng.uniform(-0.5, 0.5, 3)
                else:
                    u.v = u.v + np.tile(v, u.nodes)
        return p
    if kind == "beam":
        n = case["slabs"]
        return sg.fem_beam(seed, ny=case["ny"], nz=case["nz"], slabs=n,
                           planes=1 + 2 * n + (n + 7) // 8, length=0.5 * n / 64, vary=True,
                           corotational=case["corot"], **it)
    if kind == "cable":
        return sg.cable(seed, segments=case["segments"], **it)
    if kind == "stir":
        p = sg.stir(seed, n_side=case["side"], layers=case["layers"], **it)
        if case["pj"]:
            p.options.solver, p.options.pj_omega = "pj", 0.3
        return p
    return sg.generic(seed, n_scenes=case["scenes"], n_sub=case["subs"], n_range=(1, case["dof"]),
                      extra=case["extra"], **it)


class _State:
    pass


def _net_inputs(case, seed):
    """Weights in the range of a trained network, features of interfaces, targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng([seed, 23])
    flat = []
    for a, b in zip(NET[:-1], NET[1:]):
        flat += [rng.standard_normal(a * b) * math.sqrt(2.0 / a), 0.1 * rng.standard_normal(b)]
    w = np.concatenate(flat).astype(np.float32)
    x = torch.randn((case["batch"], NET[0]), generator=g, device="cuda")
    t = torch.randn((case["batch"], NET[-1]), generator=g, device="cuda")
    m = (torch.rand((case["batch"], NET[-1]), generator=g, device="cuda") < 0.7).float()
    return w, x, t, m


def prepare(case, seed):
    st = _State()
    st.case = case
    if case["kind"].startswith("net"):
        w, st.x, st.t, st.m = _net_inputs(case, seed)
        st.net = ws.Network(NET, stream=torch.cuda.current_stream().cuda_stream)
        st.net.set_params(w)
        st.y = torch.empty_like(st.t)
        st.grad = torch.empty(st.net.num_params, device="cuda")
        return st
    p = _problem(case, seed)
    # one large scene is spread over the whole GPU from 1024 side-rows on
    grid = 1024 if case["kind"] in ("beam", "cable", "stir") else None
    st.sim = sa.Simulation(p, stream=torch.cuda.current_stream().cuda_stream,
                           precision=sa.SIM_MIXED if case["mixed"] else sa.SIM_FP64,
                           grid_side_rows=grid)
    st.sim.launch_classes()               # lays the simulation out
    if case["kind"] == "generic":
        return st
    n = st.sim.sizes()
    n = 13 * n["bodies"] + 6 * n["nodes"]
    st.start = torch.empty(n, dtype=torch.float64, pin_memory=True)
    st.out = torch.empty(n, dtype=torch.float64, pin_memory=True)
    sa.sim_read_state(st.sim.h, st.start.data_ptr())
    return st


def run(state):
    case = state.case
    if case["kind"] == "net_infer":
        state.net.forward(state.x, state.y)
        return state.y
    if case["kind"] == "net_grad":
        state.net.gradients(state.x, state.t, state.m, state.grad)
        return state.grad
    sim = state.sim
    if case["kind"] == "generic":         # blocks given by A, b: velocities and impulses
        sim.step(case["steps"])
        v = np.concatenate([sim.scene_vhat(k) for k in range(sim.n_scenes)])
        return v.astype(np.float32) if case["mixed"] else v
    sa.sim_write_state(sim.h, state.start.data_ptr())
    sim.step(case["steps"])
    sa.sim_read_state(sim.h, state.out.data_ptr())
    return state.out.float() if case["mixed"] else state.out


def work(case):
    """Bytes: the scene's description and state in, the state out (each step's rebuilt
    quantities can stay on the chip).  Flops: the matrix K = A + beta J^T J factorised and the
    map of the constraint rows formed where they change, then per iteration the product with
    the map or with the factor, whichever is smaller."""
    if case["kind"].startswith("net"):
        par = sum(a * b for a, b in zip(NET[:-1], NET[1:]))
        io = 4 * case["batch"] * (NET[0] + NET[-1] * (1 if case["kind"] == "net_infer" else 2))
        k = 1 if case["kind"] == "net_infer" else 3
        return {"bytes": io + 4 * par * (1 if k == 1 else 2), "flops": 2.0 * k * case["batch"] * par}
    p = _problem(case, 0)
    iters = case["iters"] if "tol" not in case else 500
    byts = flops = 0.0
    for sc in p.scenes:
        m = [0] * len(sc.subs)
        for f in sc.ifs:
            if hasattr(f, "J"):
                for s in f.subs:
                    m[s] += f.rows
                    byts += 8 * f.rows * sc.subs[s].n
                continue
            r = _ROWS[f.kind]
            byts += 8 * 23
            m[f.a[0]] += r
            if f.b is not None and f.b[0] != f.a[0]:
                m[f.b[0]] += r
        for s, ms in zip(sc.subs, m):
            n = s.n
            if hasattr(s, "bodies"):
                bw, byts = min(n, 12), byts + 8 * 30 * len(s.bodies)
            elif hasattr(s, "Kv"):
                bw = int(np.max(np.abs(s.Ki - s.Kj)))
                byts += 16 * len(s.Kv) + 8 * (16 * s.nodes) + (8 * 144 * len(s.tets) if s.corot else 0)
            else:
                bw, byts = n, byts + 8 * n * n
            each = case["steps"] if not hasattr(s, "Kv") or s.corot else 0
            flops += each * (n * bw * bw + 2.0 * n * bw * ms + n * ms * ms)
            flops += case["steps"] * iters * min(2.0 * ms * ms, 4.0 * n * bw + 12.0 * ms)
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------- the same steps in plain 64-bit arithmetic

_ROWS = {sg.BALL: 3, sg.REVOLUTE: 5, sg.ANGLE_PD: 1, sg.PLANE_CONTACT: 3, sg.SPHERE_CONTACT: 3}


def _rot(q):
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                    axis=1).reshape(-1, 3, 3)


class _Flat:
    """A problem as flat arrays: bodies, nodes, subsystems, interfaces grouped by kind, and
    the side-rows of every subsystem."""

    def __init__(self, p):
        self.o = p.options
        self.subs, self.scene_of, body, node = [], [], [], []
        self.rows = 0                      # constraint rows
        self.rtype, self.k, self.al, self.mu, self.e0 = [], [], [], [], []
        self.con = []                      # first rows of contacts
        groups, self.fixed = {}, []
        self.m = []                        # side-rows per subsystem
        sr = []                            # (subsystem, local side-row, row)
        for si, sc in enumerate(p.scenes):
            base = len(self.subs)
            first = []
            for s in sc.subs:
                if hasattr(s, "bodies"):
                    first.append(len(body))
                    body += [np.concatenate([[b.m], b.I, b.p, b.q, b.v, b.w]) for b in s.bodies]
                elif hasattr(s, "Kv"):
                    first.append(len(node))
                    node += list(np.concatenate([s.x.reshape(-1, 3), s.v.reshape(-1, 3)], axis=1))
                else:
                    first.append(-1)
                self.subs.append(s)
                self.scene_of.append(si)
                self.m.append(0)

            def side(s, r):
                lo = self.m[base + s]
                self.m[base + s] += r
                sr.extend((base + s, lo + q, self.rows + q) for q in range(r))
                return lo

            for f in sc.ifs:
                if hasattr(f, "J"):
                    r = f.rows
                    self.fixed.append((self.rows, r, [(base + s, side(s, r), J) for s, J in zip(f.subs, f.J)], f.e))
                    t, k, al, mu = int(f.type), f.k, f.alpha, f.mu
                else:
                    r = _ROWS[f.kind]
                    sa_, ka = f.a
                    la = side(sa_, r)
                    na = not hasattr(sc.subs[sa_], "bodies")
                    sb, kb, lb, nb, gb = -1, 0, 0, False, -1
                    if f.b is not None and f.kind != sg.PLANE_CONTACT:
                        sb, kb = f.b
                        nb = not hasattr(sc.subs[sb], "bodies")
                        gb = first[sb] + kb
                        lb = la if sb == sa_ else side(sb, r)
                    nrm = np.asarray(f.normal, float)
                    groups.setdefault(f.kind, []).append(
                        [base + sa_, first[sa_] + ka, ka, la, na, base + sb if sb >= 0 else -1, gb, kb, lb, nb, self.rows]
                        + [*f.anchor_a, *f.anchor_b, *f.axis_a, *f.axis_b, *f.ref_a, *f.ref_b,
                           *(nrm / np.linalg.norm(nrm)), f.kp, f.kd, f.target, f.plane_z, f.mu, f.radius_a, f.radius_b])
                    t, k, al, mu = 0, 0.0, 0.0, 0.0
                    if f.kind == sg.ANGLE_PD:
                        t, k, al = 2, f.kp, f.kd / f.kp + 0.5 * self.o.h
                    elif f.kind in (sg.PLANE_CONTACT, sg.SPHERE_CONTACT):
                        t, mu = 3, f.mu
                if t == 3:
                    self.con.append(self.rows)
                for _ in range(r):
                    self.rtype.append(t)
                    self.k.append(k)
                    self.al.append(al)
                    self.mu.append(mu)
                self.rows += r
        self.body = np.array(body).reshape(-1, 17)
        self.node = np.array(node).reshape(-1, 6)
        self.groups = {k: np.array(v, dtype=np.float64) for k, v in groups.items()}
        self.n = np.array([s.n for s in self.subs])
        self.m = np.array(self.m)
        self.off = np.concatenate([[0], np.cumsum(self.m)])
        self.joff = np.concatenate([[0], np.cumsum(self.m * self.n)])
        sr = np.array(sr, dtype=np.int64).reshape(-1, 3)
        self.row_of = np.zeros(len(sr), dtype=np.int64)
        self.row_of[self.off[sr[:, 0]] + sr[:, 1]] = sr[:, 2]
        self.sub_of = np.repeat(np.arange(len(self.subs)), self.m)

    def model(self, kind, g):
        """Rows of every interface of one kind: Ja, Jb (k, r, 6) and e (k, r)."""
        h, gam = self.o.h, self.o.baumgarte
        ia, ib = g[:, 1].astype(int), g[:, 6].astype(int)
        na, nb, hasb = g[:, 4] > 0, g[:, 9] > 0, g[:, 6] >= 0
        A, B, ua, ub, ra, rb, nrm = (g[:, 11 + 3 * q:14 + 3 * q] for q in range(7))
        target, plane, r_a, r_b = g[:, 34], g[:, 35], g[:, 37], g[:, 38]
        K = len(g)

        def pose(i, is_node, has):
            R = np.tile(np.eye(3), (K, 1, 1))
            P = np.zeros((K, 3))
            s = has & ~is_node
            if s.any():
                R[s] = _rot(self.body[i[s], 7:11])
                P[s] = self.body[i[s], 4:7]
            s = has & is_node
            if s.any():
                P[s] = self.node[i[s], :3]
            return R, P

        Ra, Pa = pose(ia, na, np.ones(K, bool))
        Rb, Pb = pose(ib, nb, hasb)
        ba, bb = na[:, None], nb[:, None]
        pa = Pa + np.where(ba, 0.0, np.einsum("kij,kj->ki", Ra, A))
        pb = np.where(hasb[:, None], Pb + np.where(bb, 0.0, np.einsum("kij,kj->ki", Rb, B)), B)

        def rows(d, R, r, is_node):        # velocity of the point along d (k, 3)
            t = np.cross(r, np.einsum("kji,kj->ki", R, d))
            return np.concatenate([d, np.where(is_node[:, None], 0.0, t)], axis=1)

        nr = _ROWS[kind]
        Ja, Jb, e = np.zeros((K, nr, 6)), np.zeros((K, nr, 6)), np.zeros((K, nr))
        if kind in (sg.BALL, sg.REVOLUTE):
            for d in range(3):
                E = np.tile(np.eye(3)[d], (K, 1))
                Ja[:, d] = rows(E, Ra, A, na)
                Jb[:, d] = -rows(E, Rb, B, nb)
            e[:, :3] = gam * (pa - pb) / h
            if kind == sg.REVOLUTE:
                u = np.einsum("kij,kj->ki", Rb, ub)
                for q, t in enumerate((ra, np.cross(ua, ra))):
                    t = np.einsum("kij,kj->ki", Ra, t)
                    c = np.cross(t, u)
                    Ja[:, 3 + q, 3:] = np.einsum("kji,kj->ki", Ra, c)
                    Jb[:, 3 + q, 3:] = -np.einsum("kji,kj->ki", Rb, c)
                    e[:, 3 + q] = gam * np.sum(t * u, axis=1) / h
        elif kind == sg.ANGLE_PD:
            u, va = np.einsum("kij,kj->ki", Ra, ua), np.einsum("kij,kj->ki", Ra, ra)
            vb = np.einsum("kij,kj->ki", Rb, rb)
            th = np.arctan2(np.sum(np.cross(va, vb) * u, axis=1), np.sum(va * vb, axis=1))
            Ja[:, 0, 3:] = -np.einsum("kji,kj->ki", Ra, u)
            Jb[:, 0, 3:] = np.einsum("kji,kj->ki", Rb, u)
            e[:, 0] = th - target
        else:
            if kind == sg.PLANE_CONTACT:
                n, gap, r_b = nrm, np.sum(nrm * pa, axis=1) - plane - r_a, np.zeros(K)
            else:
                d = pa - pb
                dist = np.linalg.norm(d, axis=1)
                n = np.where(dist[:, None] > 0, d / np.where(dist > 0, dist, 1.0)[:, None], [0.0, 0.0, 1.0])
                gap = dist - r_a - r_b
            x = np.where((np.abs(n[:, 0]) > 0.9)[:, None], [0.0, 1.0, 0.0], [1.0, 0.0, 0.0])
            t1 = x - np.sum(x * n, axis=1)[:, None] * n
            t1 /= np.linalg.norm(t1, axis=1)[:, None]
            ca = A - r_a[:, None] * np.einsum("kji,kj->ki", Ra, n)
            cb = B + r_b[:, None] * np.einsum("kji,kj->ki", Rb, n)
            for q, d in enumerate((n, t1, np.cross(n, t1))):
                Ja[:, q] = rows(d, Ra, ca, na)
                if kind == sg.SPHERE_CONTACT:
                    Jb[:, q] = -rows(d, Rb, cb, nb)
            e[:, 0] = np.where(gap >= 0, gap, gam * gap) / h
        Jb[~hasb] = 0.0
        return Ja, Jb, e

    def assemble(self):
        J, e = np.zeros(self.joff[-1]), np.zeros(self.rows)
        for r0, r, sides, ee in self.fixed:
            e[r0:r0 + r] = ee
            for s, lo, M in sides:
                at = self.joff[s] + lo * self.n[s]
                J[at:at + r * self.n[s]] = np.asarray(M, float).ravel()
        for kind, g in self.groups.items():
            Ja, Jb, ee = self.model(kind, g)
            nr = _ROWS[kind]
            e[(g[:, 10].astype(int)[:, None] + np.arange(nr)).ravel()] = ee.ravel()
            for Jx, c in ((Ja, 0), (Jb, 5)):
                s, k, lo = (g[:, c + q].astype(int) for q in (0, 2, 3))
                for is_node, w in ((False, 6), (True, 3)):
                    sel = (s >= 0) & ((g[:, c + 4] > 0) == is_node)
                    if not sel.any():
                        continue
                    at = (self.joff[s[sel]] + lo[sel] * self.n[s[sel]] + w * k[sel])[:, None, None] \
                        + np.arange(nr)[None, :, None] * self.n[s[sel]][:, None, None] + np.arange(w)
                    np.add.at(J, at.ravel(), Jx[sel][:, :, :w].ravel())
        return J, e

    def blocks(self):
        """A_i and b_i of every subsystem from the present state."""
        h, g = self.o.h, np.array(self.o.gravity)
        ib = inode = 0
        for s in self.subs:
            if hasattr(s, "bodies"):
                B = self.body[ib:ib + len(s.bodies)]
                ib += len(s.bodies)
                Iw = B[:, 1:4] * B[:, 14:17]
                d = np.concatenate([np.repeat(B[:, :1], 3, axis=1), B[:, 1:4]], axis=1) * (2 / h)
                b = np.concatenate([2 / h * B[:, :1] * B[:, 11:14] + B[:, :1] * g,
                                    2 / h * Iw - np.cross(B[:, 14:17], Iw)], axis=1)
                yield np.diag(d.ravel()), b.ravel()
            elif hasattr(s, "Kv"):
                N = self.node[inode:inode + s.nodes]
                inode += s.nodes
                M = np.repeat(s.mass, 3)
                K = np.zeros((s.n, s.n))
                x, X = N[:, :3], s.X0.reshape(-1, 3)
                if not s.corot:
                    np.add.at(K, (np.asarray(s.Ki), np.asarray(s.Kj)), s.Kv)
                    f = -K @ (x - X).ravel()
                else:
                    T = np.asarray(s.tets)
                    Dm = np.swapaxes(X[T[:, 1:]] - X[T[:, :1]], 1, 2)
                    Ds = np.swapaxes(x[T[:, 1:]] - x[T[:, :1]], 1, 2)
                    U, _, Vt = np.linalg.svd(Ds @ np.linalg.inv(Dm))
                    R = U @ Vt
                    Ke = np.asarray(s.Ke).reshape(-1, 4, 3, 4, 3)
                    w = np.einsum("tji,taj->tai", R, x[T]) - X[T]
                    fe = -np.einsum("tij,taj->tai", R, np.einsum("taibj,tbj->tai", Ke, w))
                    f = np.zeros((s.nodes, 3))
                    np.add.at(f, T, fe)
                    f = f.ravel()
                    Kr = np.einsum("tij,tajbk,tlk->taibl", R, Ke, R, optimize=True).reshape(-1, 12, 12)
                    dof = (3 * T[:, :, None] + np.arange(3)).reshape(-1, 12)
                    np.add.at(K, (dof[:, :, None], dof[:, None, :]), Kr)
                yield np.diag(2 / h * M) + h / 2 * K, \
                    2 / h * M * N[:, 3:].ravel() + f + np.asarray(s.f) + M * np.tile(g, s.nodes)
            else:
                yield np.asarray(s.A, float), np.asarray(s.b, float)

    def state(self):
        return np.concatenate([self.body[:, 4:].ravel(), self.node.ravel()])


class _Map:
    """x = c + D w over all subsystems: D in batches of like sizes."""

    def __init__(self, flat, D, dev):
        self.parts = []
        order = sorted((s for s in range(len(flat.subs)) if flat.m[s]), key=lambda s: flat.m[s])
        while order:
            big = int(flat.m[order[-1]])
            part = [s for s in order if flat.m[s] * 1.3 + 4 >= big]
            order = order[:len(order) - len(part)]
            at = np.full((len(part), big), len(flat.row_of))
            M = np.zeros((len(part), big, big))
            for i, s in enumerate(part):
                m = flat.m[s]
                at[i, :m] = np.arange(flat.off[s], flat.off[s] + m)
                M[i, :m, :m] = D[s]
            self.parts.append((torch.from_numpy(at).to(dev), torch.from_numpy(M).to(dev)))

    def __call__(self, w):
        w = torch.cat([w, w.new_zeros(1)])
        x = torch.zeros_like(w)
        for at, M in self.parts:
            x[at] = torch.bmm(M, w[at][:, :, None])[:, :, 0]
        return x[:-1]


def exact(case, seed):
    if case["kind"].startswith("net"):
        return _net_exact(case, seed)
    f = _Flat(_problem(case, seed))
    o = f.o
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    pj = o.solver == "pj"
    row, scene = T(f.row_of), T(np.array(f.scene_of)[f.sub_of])
    nsc = f.scene_of[-1] + 1
    rscene = torch.zeros(f.rows, dtype=torch.int64, device=dev).scatter_(0, row, scene)
    rtype, k, al, mu = T(np.array(f.rtype)), T(np.array(f.k)), T(np.array(f.al)), T(np.array(f.mu))
    con = T(np.array(f.con, dtype=np.int64))
    lam = torch.zeros(f.rows, dtype=torch.float64, device=dev)
    z = torch.zeros(len(f.row_of), dtype=torch.float64, device=dev)
    for _ in range(case["steps"]):
        J, e = f.assemble()
        beta, D, X = np.zeros(len(f.subs)), [], []
        for s, (A, b) in enumerate(f.blocks()):
            n, m = f.n[s], f.m[s]
            Js = J[f.joff[s]:f.joff[s + 1]].reshape(m, n)
            tr = np.sum(Js * Js)
            beta[s] = 0.0 if pj else o.rho if o.beta_mode == "fixed" else np.trace(A) / tr if tr > 0 else 1.0
            Y = np.linalg.solve(A + beta[s] * Js.T @ Js, np.concatenate([Js.T, b[:, None]], axis=1))
            X.append(Y)
            D.append(Js @ Y[:, :m])
        mp = _Map(f, D, dev)
        c = T(np.concatenate([J[f.joff[s]:f.joff[s + 1]].reshape(f.m[s], f.n[s]) @ X[s][:, -1] for s in range(len(f.subs))]))
        e_ = T(e)
        if o.warm != "prev":
            lam, z = torch.zeros_like(lam), torch.zeros_like(z)
        add = lambda v: torch.zeros_like(lam).index_add_(0, row, v)  # noqa: E731

        def cone(l0, l1, l2):
            l0 = l0.clamp(min=0.0)
            t = torch.sqrt(l1 * l1 + l2 * l2)
            q = torch.where(t > mu[con] * l0, mu[con] * l0 / t.clamp(min=1e-300), torch.ones_like(t))
            return l0, l1 * q, l2 * q

        if pj:
            diag = T(np.concatenate([np.diag(d) for d in D]))
            dl = add(diag)
            dl[con + 1] = dl[con + 2] = torch.maximum(dl[con + 1], dl[con + 2])
            om = o.pj_omega
            for _ in range(o.max_iters):
                x = add(c + mp(lam[row]))
                new = lam - om * (x + e_) / dl
                soft = lam + om * (-k * (e_ + al * (x - dl * lam)) / (1 + k * al * dl) - lam)
                new = torch.where(rtype == 2, soft, torch.where(rtype == 1, new.clamp(min=0.0), new))
                new[con], new[con + 1], new[con + 2] = cone(new[con], new[con + 1], new[con + 2])
                lam = new
            last = lam[row]
            z = c + mp(last)
        else:
            bt = T(beta[f.sub_of])
            s = add(1.0 / bt)
            w, last = bt * z + lam[row], None
            on = torch.ones(nsc, dtype=torch.bool, device=dev)
            last = w.clone()
            for _ in range(o.max_iters):
                x = c + mp(w)
                y = bt * x - lam[row]
                q = add(y / bt)
                new = torch.where(rtype == 2, -k * (e_ + al * q) / (1 + s * al * k), -(q + e_) / s)
                new = torch.where(rtype == 1, new.clamp(min=0.0), new)
                new[con], new[con + 1], new[con + 2] = cone(new[con], new[con + 1], new[con + 2])
                zn = (y + new[row]) / bt
                live = on[scene]
                last = torch.where(live, w, last)
                if o.tol_primal > 0:
                    r = torch.maximum((x - zn).abs(), (zn - z).abs())
                    over = torch.zeros(nsc, dtype=torch.float64, device=dev).scatter_reduce_(0, scene, r, "amax")
                lam = torch.where(on[rscene], new, lam)
                z = torch.where(live, zn, z)
                w = torch.where(live, y + 2 * new[row], w)
                if o.tol_primal > 0:
                    on = on & (over > o.tol_primal)
                    if not bool(on.any()):
                        break
        wl, vs = last.cpu().numpy(), []
        for s in range(len(f.subs)):
            vs.append(X[s][:, -1] + X[s][:, :-1] @ wl[f.off[s]:f.off[s + 1]])
        ib = inode = 0
        for s, v in zip(f.subs, vs):
            if hasattr(s, "bodies"):
                B = f.body[ib:ib + len(s.bodies)]
                ib += len(s.bodies)
                v = v.reshape(-1, 6)
                B[:, 4:7] += o.h * v[:, :3]
                B[:, 11:17] = 2 * v - B[:, 11:17]
                a = o.h * v[:, 3:]
                th = np.linalg.norm(a, axis=1)[:, None]
                sn = np.where(th > 0, np.sin(th / 2) / np.where(th > 0, th, 1.0), 0.0)
                d, q = np.concatenate([np.cos(th / 2), a * sn], axis=1), B[:, 7:11].copy()
                B[:, 7] = q[:, 0] * d[:, 0] - np.sum(q[:, 1:] * d[:, 1:], axis=1)
                B[:, 8:11] = q[:, :1] * d[:, 1:] + d[:, :1] * q[:, 1:] + np.cross(q[:, 1:], d[:, 1:])
                B[:, 7:11] /= np.linalg.norm(B[:, 7:11], axis=1)[:, None]
            elif hasattr(s, "Kv"):
                N = f.node[inode:inode + s.nodes]
                inode += s.nodes
                v = v.reshape(-1, 3)
                N[:, :3] += o.h * v
                N[:, 3:] = 2 * v - N[:, 3:]
    return np.concatenate(vs) if case["kind"] == "generic" else f.state()


def _net_exact(case, seed):
    w, x, t, m = _net_inputs(case, seed)
    a, par, off = [x.double()], [], 0
    for i, j in zip(NET[:-1], NET[1:]):
        W = torch.from_numpy(w[off:off + i * j]).double().reshape(i, j).cuda()
        b = torch.from_numpy(w[off + i * j:off + i * j + j]).double().cuda()
        par += [W.requires_grad_(), b.requires_grad_()]
        off += i * j + j
    grad = case["kind"] == "net_grad"
    with torch.set_grad_enabled(grad):
        y = a[0]
        for q in range(4):
            y = y @ par[2 * q] + par[2 * q + 1]
            if q < 3:
                y = torch.nn.functional.gelu(y)
        if not grad:
            return y.cpu().numpy()
        (0.5 * (m * (y - t) ** 2).sum() / case["batch"]).backward()
    return np.concatenate([v.grad.reshape(-1).cpu().numpy() for v in par])

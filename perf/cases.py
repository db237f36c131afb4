"""The measured work of this framework: its per-timestep solve and its adjoint through the
public entry points, from one world to a full batch.

A case names the scene, the number of worlds, the element type and the operation:

  step       one forward step, nothing recorded (plain simulation)
  adjoint    one recorded step and its adjoint in the paper's mode (one link of every
             gradient)
  params     the same with the gradients of the servo gains, masses, inertias and mu
  exact      the same with the exact implicit-function adjoint
  pcr        the same with the matrix-free conjugate-residual solver, 16 iterations
  list       a recorded step and its adjoint of a selected subset of the worlds of a pool
             (what the serving loop issues every tick)
  noalloc    the allocation-free step and adjoint
  chunk      a captured graph of ten recorded steps and their adjoints
  rollout    a checkpointed rollout of a horizon, its loss and the gradient of the control
             splines (the body of an optimisation iteration)

The worlds stand where a rollout meets them: robots on the flat approach, at the
obstacle's face and on its top (or on the terrain), rolling at up to the speed that the
servo targets ask for, with the static wheel loads as the multipliers carried over from
the step before; boxes just above, in and a little through their contacts, tilted and
sliding.
"""
import math

import numpy as np
import torch

from paper_2609_08800_gb300 import scenes as S
from paper_2609_08800_gb300 import spline as SP
from paper_2609_08800_gb300 import tune
from paper_2609_08800_gb300.autograd import CudaEngine, rollout
from paper_2609_08800_gb300.graphs import ChunkGraph
from paper_2609_08800_gb300.ostrich import ADJ_EXACT, Context, ostrich_step_adjoint_noalloc

H = 0.1            # time step (s), as in every workload of this repository
SEGMENT = 10       # checkpoint segment of the rollouts, steps of a captured chunk
KNOTS = 8          # knots of a wheel's control spline
GRAVITY = 9.81


def listed():
    return [
        # a real-time control loop around one robot: a step and its gradient, latency alone
        dict(name="robot_1", scene="robot_box", op="adjoint", worlds=1, dtype="f32", tuned=False, horizon=1),
        # a handful of boxes in double precision: a check of gradients, a small study
        dict(name="box_37_f64", scene="box", op="adjoint", worlds=37, dtype="f64", tuned=False, horizon=1),
        # the smallest scene over a batch: dropped boxes, one contact group, no joints
        dict(name="box_4096", scene="box", op="adjoint", worlds=4096, dtype="f32", tuned=True, horizon=1),
        # plain simulation of an odd number of robots on the plane, default settings
        dict(name="plane_1001_forward", scene="robot_plane", op="step", worlds=1001, dtype="f32", tuned=False, horizon=1),
        # the main path: the wheeled robot over the box obstacle, full batch
        dict(name="robot_8192", scene="robot_box", op="adjoint", worlds=8192, dtype="f32", tuned=True, horizon=1),
        # robots on the mesh terrain: the largest contact groups, truncated pull-back
        dict(name="terrain_2048", scene="terrain", op="adjoint", worlds=2048, dtype="f32", tuned=True, horizon=1),
        # the main path in double precision
        dict(name="robot_304_f64", scene="robot_box", op="adjoint", worlds=304, dtype="f64", tuned=True, horizon=1),
        # gradients without the frozen friction weight's bias
        dict(name="robot_exact_2048", scene="robot_box", op="exact", worlds=2048, dtype="f32", tuned=True, horizon=1),
        # system identification: gradients of the physical parameters
        dict(name="robot_params_1537", scene="robot_box", op="params", worlds=1537, dtype="f32", tuned=True, horizon=1),
        # the paper's own linear solver at its 16 x 16 iterations
        dict(name="robot_pcr_512", scene="robot_box", op="pcr", worlds=512, dtype="f32", tuned=True, horizon=1),
        # a tick of the serving loop: a scattered subset of a pool's worlds
        dict(name="serve_tick_700", scene="robot_box", op="list", worlds=700, dtype="f32", tuned=True, horizon=1),
        # an optimisation iteration: rollout with checkpoints, loss, gradient of the splines
        dict(name="optimise_1024x20", scene="robot_box", op="rollout", worlds=1024, dtype="f32", tuned=True, horizon=20),
    ]


# worlds of the largest drawn case of each (operation, element type): none costs more than
# the largest listed one
_MOST = {("step", "f32"): 8192, ("adjoint", "f32"): 8192, ("params", "f32"): 8192, ("exact", "f32"): 3072,
         ("pcr", "f32"): 1536, ("list", "f32"): 4096, ("noalloc", "f32"): 1600, ("chunk", "f32"): 512,
         ("rollout", "f32"): 768, ("step", "f64"): 768, ("adjoint", "f64"): 640}


def draw(rng):
    op, dtype = rng.choice(sorted(_MOST))
    if op in ("step", "adjoint"):
        scene = rng.choice(["box", "robot_plane", "robot_box", "robot_box", "terrain"])
    elif op in ("noalloc", "params"):
        scene = rng.choice(["box", "robot_plane", "robot_box"])
    else:
        scene = "robot_box"
    most = _MOST[(op, dtype)]
    if scene == "terrain":
        most = most // 4
    worlds = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    horizon = {"rollout": rng.randint(11, 24), "chunk": SEGMENT}.get(op, 1)
    return dict(scene=scene, op=op, worlds=max(1, worlds), dtype=dtype, tuned=rng.random() < 0.7, horizon=horizon)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_SCENES = {}


def _scene(name):
    """The scene data, made once (the terrain's heightmap is the repository's seeded one)."""
    if name not in _SCENES:
        _SCENES[name] = {"box": S.box_drop_scene, "robot_plane": S.robot_plane_scene, "robot_box": S.robot_box_scene,
                         "terrain": S.terrain_scene}[name]()
    return _SCENES[name]


def _config(case):
    cfg = S.SolverConfig(tol=1e-4 if case["dtype"] == "f32" else 1e-5)
    if case["scene"] == "terrain":
        cfg.pullback = S.PULLBACK_TRUNCATED
    if case["op"] == "pcr":
        cfg.linear_solver, cfg.precond, cfg.pcr_iters = S.LIN_PCR, S.PC_JACOBI, 16
    return cfg


def _box_states(scene, W, rng):
    """Boxes from 2 cm above to 6 mm into the plane, tilted by up to 0.2 rad about x, sliding."""
    s = np.zeros((scene.n_state, W))
    half = np.array(scene.bodies[0].half_extents)
    ang = rng.uniform(-0.2, 0.2, W) * (rng.random(W) < 0.5)
    low = half[2] * np.cos(ang) + half[1] * np.abs(np.sin(ang))       # centre height over the lowest corner
    s[0], s[1], s[2] = rng.uniform(-1, 1, W), rng.uniform(-1, 1, W), low + rng.uniform(-0.006, 0.02, W)
    s[3], s[4] = np.cos(ang / 2), np.sin(ang / 2)
    s[7], s[8] = rng.uniform(0.0, 1.0, W), rng.uniform(-0.3, 0.3, W)
    return s


def _robot_states(scene, W, rng):
    """Robots placed as the repository's generators place them (half on the flat approach, a
    quarter at the obstacle's face, a quarter on its top; anywhere on the plane or the
    terrain), rolling without slip at up to 5 rad/s, the wheels loaded with the robot's weight."""
    nb = scene.n_bodies
    s = np.zeros((scene.n_state, W))
    r = S.ROBOT_WHEEL_RADIUS
    kind = scene.env.kind
    if kind == S.ENV_HEIGHTMAP:
        s[:7 * nb] = S.terrain_states(scene, W, seed=int(rng.integers(1 << 30)))[:7 * nb]
        s[2:7 * nb:7] -= 0.012                                        # standing on the terrain
        psi = 2.0 * np.arctan2(s[6], s[3])
        feature = np.zeros(W, dtype=int)
    else:
        psi = rng.uniform(-0.3, 0.3, W)
        x, z = rng.uniform(-0.6, 0.3, W), np.full(W, S.ROBOT_CHASSIS_Z)
        feature = np.zeros(W, dtype=int)
        if kind == S.ENV_BOX:
            x0, x1, _, _, top = scene.env.box
            u = rng.random(W)
            face, on = (u >= 0.5) & (u < 0.75), u >= 0.75
            psi = np.where(face, 0.0, psi)
            x = np.where(face, x0 - 0.25 - r - rng.uniform(0.0, 0.01, W), x)
            x = np.where(on, rng.uniform(x0 + 0.45, x1 - 0.45, W), x)
            z = np.where(on, z + top, z)
            feature = on.astype(int)
        c, n = np.cos(psi), np.sin(psi)
        for b in range(nb):
            ox, oy = (0.0, 0.0) if b == 0 else S.ROBOT_WHEEL_OFFSETS[b - 1][:2]
            s[7 * b], s[7 * b + 1], s[7 * b + 2] = x + c * ox - n * oy, n * ox + c * oy, z
            s[7 * b + 3], s[7 * b + 6] = np.cos(psi / 2), np.sin(psi / 2)
    spin = rng.uniform(-4.0, 5.0, W)
    for b in range(nb):
        u = 7 * nb + 6 * b
        s[u], s[u + 1] = r * spin * np.cos(psi), r * spin * np.sin(psi)
        if b:
            s[u + 3], s[u + 4] = -spin * np.sin(psi), spin * np.cos(psi)
    if kind != S.ENV_HEIGHTMAP:
        nf = scene.features_per_rim()
        load = sum(b.mass for b in scene.bodies) * GRAVITY / (2 * (nb - 1))
        for rim in range(2 * (nb - 1)):
            s[scene.contact_lam_index + 3 * (rim * nf + feature), np.arange(W)] = load
    return s


def _inputs(case, seed):
    """States, servo targets and the cotangent of the next state (host, double)."""
    scene, rng = _scene(case["scene"]), np.random.default_rng(seed)
    W = case["worlds"]
    s = (_box_states if case["scene"] == "box" else _robot_states)(scene, W, rng)
    ctl = rng.uniform(-5.0, 5.0, (scene.n_servos, W))
    g = np.zeros_like(s)                    # of |p_xy - (3, 0)|^2 of the first body, as the optimisation takes it
    g[0], g[1] = 2.0 * (s[0] - 3.0), 2.0 * s[1]
    return scene, s, ctl, g, rng


def prepare(case, seed):
    scene, s, ctl, g, rng = _inputs(case, seed)
    op, W, dt = case["op"], case["worlds"], torch.float64 if case["dtype"] == "f64" else torch.float32
    cfg = _config(case)

    def dev(a):
        return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")

    st = dict(op=op, scene=scene, cfg=cfg, s=dev(s), ctl=dev(ctl) if scene.n_servos else None, g=dev(g))
    if op == "noalloc":
        st.update(out=torch.empty_like(st["s"]), ds=torch.empty_like(st["s"]),
                  dctl=torch.empty_like(st["ctl"]) if scene.n_servos else None)
        return st
    if op == "rollout":
        T = case["horizon"]
        st["eng"] = CudaEngine(scene, cfg, W, H, slots=SEGMENT, dtype=case["dtype"])
        if case["tuned"]:
            tune.apply(st["eng"].ctx)
        st["basis"] = dev(SP.basis(T, KNOTS, H))
        st["knots"] = dev(rng.uniform(-5.0, 5.0, (W, scene.n_servos, KNOTS))).requires_grad_(True)
        return st
    pool = W if op != "list" else W + W // 2 + 1
    slots = {"step": 0, "list": 2, "chunk": SEGMENT}.get(op, 1)
    ctx = Context(scene, cfg, pool, dtype=case["dtype"], tape_slots=slots)
    if case["tuned"]:
        tune.apply(ctx)
    st["ctx"] = ctx
    if op == "list":
        cols = np.sort(rng.permutation(pool)[:W])
        for key, a in (("s", s), ("ctl", ctl), ("g", g)):
            wide = np.zeros((a.shape[0], pool))
            wide[:, cols] = a
            st[key] = dev(wide)
        st["cols"] = torch.tensor(cols, dtype=torch.int32, device="cuda")
        st["slots"] = torch.tensor(rng.integers(0, 2, W), dtype=torch.int32, device="cuda")
        st.update(out=torch.zeros_like(st["s"]), ds=torch.zeros_like(st["s"]), dctl=torch.zeros_like(st["ctl"]))
    elif op == "chunk":
        knots = rng.uniform(-5.0, 5.0, (W, scene.n_servos, KNOTS))
        st["ctls"] = dev(np.einsum("tk,wjk->tjw", SP.basis(10 * SEGMENT, KNOTS, H)[:SEGMENT], knots))
        st["graph"] = ChunkGraph(ctx, SEGMENT, H)
    elif op == "exact":
        ctx.set_adjoint_mode(ADJ_EXACT)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    op = st["op"]
    if op == "noalloc":
        ostrich_step_adjoint_noalloc(st["scene"], st["cfg"], st["s"].shape[1], st["s"], st["ctl"], H, st["out"], st["g"],
                                     st["ds"], st["dctl"])
        return dict(state=st["out"], dstate=st["ds"], dctl=st["dctl"])
    if op == "rollout":
        st["knots"].grad = None
        controls = torch.einsum("tk,wjk->tjw", st["basis"], st["knots"]).contiguous()
        traj = rollout(st["s"], controls, st["eng"], segment=SEGMENT)
        loss = (traj[-1][0] - 3.0) ** 2 + traj[-1][1] ** 2
        torch.where(torch.isfinite(loss), loss, torch.zeros_like(loss)).sum().backward()
        return dict(traj=traj.detach(), loss=loss.detach(), dknots=st["knots"].grad)
    ctx = st["ctx"]
    if op == "list":
        ctx.ostrich_step_list(st["s"], st["ctl"], H, st["out"], st["cols"], st["slots"])
        ctx.ostrich_adjoint_list(st["g"], H, st["ds"], st["cols"], st["slots"], st["dctl"])
        return dict(state=st["out"], dstate=st["ds"], dctl=st["dctl"])
    if op == "chunk":
        states, grads, dctl = st["graph"].replay(st["s"], st["ctls"], st["g"])
        return dict(states=states, grads=grads, dctl=dctl)
    r = ctx.step(st["s"], st["ctl"], H, tape_slot=-1 if op == "step" else 0)
    out = {k: r[k] for k in ("state", "impulses", "ids", "status")}
    if op == "params":
        out.update(zip(("dstate", "dctl", "dkp", "dmass", "dinertia", "dmu"),
                       ctx.adjoint_params(0, st["g"], H, with_mu=True)))
    elif op != "step":
        out["dstate"], out["dctl"] = ctx.adjoint(0, st["g"], H)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _world_flops(scene):
    """Operations of one world's Newton iteration with its usual contacts (a box on four
    corners, every rim of a robot on one face): rows and residual, the block-arrowhead
    matrix, its factor and a solve."""
    sep = 5 * len(scene.joints) + scene.n_servos
    groups = [12] if not scene.joints else [6] * (scene.n_bodies - 1)
    m = sum(groups) + sep
    return (250 * m + sum(6 * p * (p + 1) + 72 * p for p in groups) + 12 * sep * (sep + 1)
            + sum(p ** 3 / 3 + 6 * p * p + 36 * p for p in groups) + sep ** 3 / 3
            + 2 * (sum(p * p for p in groups) + sep * sep) + 24 * sum(groups))


def work(case):
    scene, op, W, T = _scene(case["scene"]), case["op"], case["worlds"], case["horizon"]
    e = 8 if case["dtype"] == "f64" else 4
    ns, nv = scene.n_state, scene.n_servos
    newton = 4 if case["scene"] == "box" else 10          # iterations of an ordinary step
    fwd = newton * _world_flops(scene)
    adj = 3 * _world_flops(scene)                          # one solve with refinement and the pull-back
    bytes_fwd = e * (2 * ns + nv)
    bytes_adj = e * (2 * ns + nv)
    if op in ("step", "adjoint", "params", "exact", "pcr"):
        bytes_fwd += e * scene.m_max + 4 * (scene.n_slots + 1)
    if op == "step":
        return dict(bytes=W * bytes_fwd, flops=W * fwd)
    if op == "params":
        bytes_adj += e * (nv + 4 * scene.n_bodies + 1)
    if op == "exact":
        adj = 3 * adj
    if op in ("rollout", "chunk"):
        # every step once, its adjoint once; a rollout also writes its trajectory and
        # reads and writes the splines
        more = e * 2 * KNOTS * nv if op == "rollout" else e * T * ns
        return dict(bytes=W * (e * (T + 1) * ns + more), flops=W * T * (fwd + adj))
    return dict(bytes=W * (bytes_fwd + bytes_adj), flops=W * (fwd + adj))


# ---------------------------------------------------------------------------
# 64-bit values (boxes on the plane: every step of theirs is solved)
# ---------------------------------------------------------------------------
def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _rot(q):
    """Rotation matrices of unnormalised quaternions (w, x, y, z): [W, 3, 3]."""
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)


def _advance(q, u):
    """Backward-Euler positions: p + h v, quat + h/2 (0, w) (x) quat (not normalised)."""
    qw, qv, om = q[:, 3:4], q[:, 4:], u[:, 3:]
    return torch.cat([q[:, :3] + H * u[:, :3], qw - 0.5 * H * (om * qv).sum(-1, keepdim=True),
                      qv + 0.5 * H * (om * qw + _cross(om, qv))], -1)


class _Box:
    """The box-on-plane step in 64 bits over a batch: residual rows, Newton, adjoint."""

    def __init__(self, scene, cfg, s):
        b = scene.bodies[0]
        self.cfg, self.mu, self.m = cfg, scene.mu, b.mass
        self.I = torch.tensor(b.inertia, dtype=torch.float64, device=s.device)
        self.corner = torch.tensor([[b.half_extents[a] * (1 if k >> a & 1 else -1) for a in range(3)] for k in range(8)],
                                   dtype=torch.float64, device=s.device)
        self.q, self.u, self.lam = s[:, :7], s[:, 7:13], s[:, 13:].reshape(-1, 8, 3)
        self.Iw, self.f = self.body(self.q, self.u)
        self.Iwi = torch.linalg.inv(self.Iw)
        R = _rot(self.q[:, 3:])
        lev = torch.einsum("wij,kj->wki", R, self.corner)
        vp = self.u[:, None, :3] + _cross(self.u[:, None, 3:].expand_as(lev), lev)
        app = vp[..., 2] - H * GRAVITY
        # activation is decided in single precision: the set is the one a correctly
        # rounded predicate gives, away from its threshold
        self.on = self.q[:, None, 2] + lev[..., 2] + H * app.clamp(max=0.0) < cfg.margin
        a = _cross(lev, torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=s.device).expand_as(lev))
        self.what = 1.0 / self.m + torch.einsum("wki,wij,wkj->wk", a, self.Iwi, a)

    def body(self, q, u):
        R = _rot(q[:, 3:])
        Iw = torch.einsum("wij,j,wkj->wik", R, self.I, R)
        gy = _cross(u[:, 3:], torch.einsum("wij,wj->wi", Iw, u[:, 3:]))
        lin = torch.zeros_like(gy)
        lin[:, 2] = -self.m * GRAVITY
        return Iw, torch.cat([lin, -gy], -1)

    def minv(self, v):
        return torch.cat([v[..., :3] / self.m, torch.einsum("wij,w...j->w...i", self.Iwi, v[..., 3:])], -1)

    def jac(self, q, u):
        """Rows (normal, two tangents) of the eight corners, [W, 8, 3, 6], and the gaps."""
        qp = _advance(q, u)
        lev = torch.einsum("wij,kj->wki", _rot(qp[:, 3:]), self.corner)
        D = torch.tensor([[0., 0., 1.], [1., 0., 0.], [0., 1., 0.]], dtype=torch.float64, device=q.device)
        lev4, d4 = torch.broadcast_tensors(lev[:, :, None], D[None, None])
        a, om = _cross(lev4, d4), u[:, None, None, 3:]
        a = (a + 0.5 * H * _cross(a, om.expand_as(a))) / (1.0 + 0.25 * H * H * (om * om).sum(-1, keepdim=True))
        return torch.cat([d4, a], -1), qp[:, None, 2] + lev[..., 2], qp

    def rows(self, u, lam):
        c, on = self.cfg, self.on
        J, gap, _ = self.jac(self.q, u)
        J = J * on[..., None, None]
        eps, kap, hw = c.eps_fb, c.kappa, H * self.what
        vel = torch.einsum("wkrc,wc->wkr", J, u)
        ln, lf = lam[..., 0], lam[..., 1:]
        a, b = gap / H + kap * ln, hw * ln
        s = torch.sqrt(a * a + b * b + eps * eps)
        phi = torch.where(a + b > 0, (2 * a * b - eps * eps) / (a + b + s), a + b - s)
        fa = torch.where(a > 0, (b * b + eps * eps) / (s * (s + a)), 1 - a / s)
        fb = torch.where(b > 0, (a * a + eps * eps) / (s * (s + b)), 1 - b / s)
        scl = fa.clamp(min=1e-12)
        vt = torch.sqrt((vel[..., 1:] ** 2).sum(-1) + eps * eps)
        lfn = torch.sqrt((lf ** 2).sum(-1) + eps * eps)
        lnp = ln.clamp(min=0.0)
        g = hw * (self.mu * lnp - lfn)
        sg = torch.sqrt(vt * vt + g * g + eps * eps)
        num = torch.where(g > 0, (vt * vt + eps * eps) / (sg + g), sg - g)
        den = (self.mu * lnp).clamp(min=1e-12)
        Wf = num / den
        rf = vel[..., 1:] + (Wf + kap)[..., None] * lf
        r2 = torch.cat([phi[..., None], rf * (hw / (hw + Wf))[..., None]], -1) * on[..., None]
        rhat = torch.cat([(phi / scl)[..., None], rf], -1) * on[..., None]
        C = torch.zeros(*ln.shape, 3, 3, dtype=torch.float64, device=u.device)
        C[..., 0, 0] = kap + hw * fb / scl
        e = lf / lfn[..., None]
        rho = torch.where(num > 0, num / sg * hw * lfn / den, torch.zeros_like(num))
        C[..., 1:, 1:] = (Wf + kap)[..., None, None] * torch.eye(2, dtype=torch.float64, device=u.device) \
            + rho[..., None, None] * e[..., :, None] * e[..., None, :]
        eye = torch.eye(3, dtype=torch.float64, device=u.device)
        C = torch.where(on[..., None, None], C, eye)
        M6 = torch.cat([self.m * (u - self.u)[:, :3], torch.einsum("wij,wj->wi", self.Iw, (u - self.u)[:, 3:])], -1)
        rdyn = M6 - H * self.f - H * torch.einsum("wkrc,wkr->wc", J, lam)
        merit = (self.minv(rdyn) ** 2).sum(-1) + (r2 ** 2).sum((-1, -2))
        return J, rhat, C, rdyn, merit

    def matrix(self, J, C):
        W = J.shape[0]
        Jf = J.reshape(W, 24, 6)
        A = H * torch.einsum("wic,wjc->wij", Jf, self.minv(Jf))
        m = (3 * self.on.sum(-1)).clamp(min=1)
        delta = self.cfg.delta_rel * A.diagonal(dim1=1, dim2=2).sum(-1) / m
        for k in range(8):
            A[:, 3 * k:3 * k + 3, 3 * k:3 * k + 3] += C[:, k]
        return A + delta[:, None, None] * torch.eye(24, dtype=torch.float64, device=J.device)

    def clamp(self, lam):
        rad = self.mu * lam[..., 0].clamp(min=0.0)
        n = lam[..., 1:].norm(dim=-1)
        f = torch.where(n > rad, rad / n.clamp(min=1e-300), torch.ones_like(n))
        return torch.cat([lam[..., :1], lam[..., 1:] * f[..., None]], -1) * self.on[..., None]

    def solve(self):
        u = self.u + H * self.minv(self.f)
        lam = self.clamp(self.lam)
        for _ in range(80):
            J, rhat, C, rdyn, merit = self.rows(u, lam)
            if bool((merit < 1e-22).all()):
                break
            W = u.shape[0]
            rhs = torch.einsum("wkrc,wc->wkr", J, self.minv(rdyn)) - rhat
            dl = torch.linalg.solve(self.matrix(J, C), rhs.reshape(W, 24)).reshape(W, 8, 3)
            go = (merit >= 1e-22)[:, None]
            u = torch.where(go, u + self.minv(H * torch.einsum("wkrc,wkr->wc", J, dl) - rdyn), u)
            lam = torch.where(go[..., None], self.clamp(lam + dl), lam)
        return u, lam, float(merit.max())

    def adjoint(self, u, lam, g):
        W = u.shape[0]
        J, _, C, _, _ = self.rows(u, lam)
        q = self.q.clone().requires_grad_(True)
        um = self.u.clone().requires_grad_(True)
        u_ = u.clone().requires_grad_(True)

        def forward_pose(q, u):
            qp = _advance(q, u)
            return torch.cat([qp[:, :3], qp[:, 3:] / qp[:, 3:].norm(dim=-1, keepdim=True)], -1)

        gu = g[:, 7:13] + torch.autograd.grad((forward_pose(self.q, u_) * g[:, :7]).sum(), u_)[0]
        Jf = J.reshape(W, 24, 6)
        rhs = -H * torch.einsum("wic,wc->wi", Jf, self.minv(gu))
        wl = torch.linalg.solve(self.matrix(J, C), rhs)
        wu = -self.minv(gu + torch.einsum("wic,wi->wc", Jf, wl))
        wl = wl.reshape(W, 8, 3) * self.on[..., None]
        # the explicit partials along the step's inputs, u+ and lambda+ held
        Iw, f = self.body(q, um)
        dyn = torch.cat([self.m * (u - um)[:, :3], torch.einsum("wij,wj->wi", Iw, (u - um)[:, 3:])], -1) - H * f
        Jq, gap, _ = self.jac(q, u)
        Jq = Jq * self.on[..., None, None]
        vel = torch.einsum("wkrc,wc->wkr", Jq, u)
        psi = (forward_pose(q, u) * g[:, :7]).sum() + (wu * dyn).sum() \
            + (wl[..., 0] * gap).sum() / H + (wl[..., 1:] * vel[..., 1:]).sum() \
            - H * (lam * torch.einsum("wkrc,wc->wkr", Jq, wu)).sum()
        dq, du = torch.autograd.grad(psi, (q, um))
        return torch.cat([dq, du, torch.zeros(W, 24, dtype=torch.float64, device=u.device)], -1)


def exact(case, seed):
    """64-bit values of the boxes' step and adjoint.  A robot's step often ends on its budget
    (a sliding, lightly loaded wheel), and what it returns there is its best iterate and no
    solution: such outputs have no value of their own in 64 bits."""
    if case["scene"] != "box" or case["op"] not in ("step", "adjoint", "noalloc"):
        return None
    scene, s, _, g, _ = _inputs(case, seed)
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    s, g = (torch.tensor(a, dtype=dt, device="cuda").double().T.contiguous() for a in (s, g))
    box = _Box(scene, _config(case), s)
    u, lam, merit = box.solve()
    if not merit < 1e-16:
        return None
    qp = _advance(box.q, u)
    qp = torch.cat([qp[:, :3], qp[:, 3:] / qp[:, 3:].norm(dim=-1, keepdim=True)], -1)
    lam = lam.reshape(-1, 24)
    state = torch.cat([qp, u, lam], -1).T.contiguous()
    if case["op"] == "noalloc":
        return dict(state=state, dstate=box.adjoint(u, lam.reshape(-1, 8, 3), g).T.contiguous(), dctl=None)
    out = dict(state=state, impulses=H * lam.T.contiguous(), ids=None, status=None)
    if case["op"] == "adjoint":
        out["dstate"], out["dctl"] = box.adjoint(u, lam.reshape(-1, 8, 3), g).T.contiguous(), None
    return out

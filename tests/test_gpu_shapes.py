"""Block sizes and launch shapes at the edges of the kernels' variants, against the oracle.

* vehicles of 5, 6 and 7 wheels: separators of 30, 36 and 42 rows, on both sides of the 32
  rows one warp's registers hold (their factor's order and that of the whole CTA);
* hinged boxes with every corner active: contact groups of 24 rows (one block per warp; the
  usual ones go two to a warp up to 16 rows), two groups sharing the joint's rows;
* few worlds run with more warps each (normals and friction in different ones), many with the
  context's threads: the results of a world are bit-identical either way.

Tolerances are those of the parity tests of the same precision (test_gpu_parity.py): FP64
1e-7 / 1e-6 / 1e-6, FP32 1e-4 / 1e-3 / 1e-3 for worlds whose iterate solves the step.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_08800_gb300 import scenes as S  # noqa: E402
from tests.test_gpu_parity import _compare, _hinged_states, ostrich  # noqa: E402,F401
from tests.test_oracle_pins import hinged_boxes_scene  # noqa: E402

H = 0.1


def vehicle_scene(n_wheels):
    """A chassis on n wheels in two staggered rows on the plane, every axle with a servo."""
    bodies = [S.Body(mass=20.0, inertia=S._box_inertia(20.0, 1.2, 0.4, 0.15))]
    joints, offs = [], []
    for i in range(n_wheels):
        off = (0.45 - 0.9 * i / (n_wheels - 1), 0.25 if i % 2 else -0.25, 0.0)
        bodies.append(S.Body(mass=1.0, inertia=S._cyl_inertia_y(1.0, 0.15, 0.08), shape=S.SHAPE_WHEEL, radius=0.15,
                             half_width=0.04))
        joints.append(S.Joint(parent=0, child=i + 1, anchor_parent=off, anchor_child=(0.0, 0.0, 0.0), kp=50.0))
        offs.append(off)
    return S.Scene("vehicle", bodies, joints, S.Env(S.ENV_PLANE), 0.9), offs


def vehicle_states(sc, offs, W, seed):
    rng = np.random.default_rng(seed)
    st = np.zeros((sc.n_state, W))
    nb = sc.n_bodies
    for w in range(W):
        x, psi, v = rng.uniform(-1, 1), rng.uniform(-0.3, 0.3), rng.uniform(-0.3, 0.3)
        c, s = np.cos(psi), np.sin(psi)
        for b in range(nb):
            ox, oy = (0.0, 0.0) if b == 0 else offs[b - 1][:2]
            st[7 * b:7 * b + 7, w] = (x + c * ox - s * oy, s * ox + c * oy, 0.15, np.cos(psi / 2), 0, 0, np.sin(psi / 2))
            st[7 * nb + 6 * b:7 * nb + 6 * b + 2, w] = v * c, v * s
            if b:
                st[7 * nb + 6 * b + 3:7 * nb + 6 * b + 5, w] = -v / 0.15 * s, v / 0.15 * c
    return st


@pytest.mark.parametrize("n_wheels,dtype,threads", [(5, "f64", 64), (6, "f64", 32), (6, "f64", 64), (7, "f64", 64),
                                                    (7, "f64", 128), (5, "f32", 64), (6, "f32", 64), (7, "f32", 128)])
def test_separator_sizes_match_oracle(ostrich, n_wheels, dtype, threads):  # noqa: F811
    sc, offs = vehicle_scene(n_wheels)
    W = 12
    st = vehicle_states(sc, offs, W, n_wheels)
    ub = S.random_controls(sc.n_servos, W, seed=n_wheels, low=-2, high=2)
    g = np.random.default_rng(n_wheels).normal(size=st.shape)
    g[13 * sc.n_bodies:] = 0
    if dtype == "f64":
        _compare(sc, S.SolverConfig(budget=60, tol=1e-9), ostrich, st, ub, H, "f64", 1e-7, 1e-6, 1e-6, 0.5, grads=g,
                 threads=threads)
    else:
        _compare(sc, S.SolverConfig(budget=40), ostrich, st, ub, H, "f32", 1e-4, 1e-3, 1e-3, 0.5, grads=g,
                 oracle_cfg=S.SolverConfig(budget=60, tol=1e-8), floor=3e-4, threads=threads, tol_grad_exact=3e-3)


@pytest.mark.parametrize("threads", [32, 64, 128])
def test_full_contact_groups_match_oracle(ostrich, threads):  # noqa: F811
    sc = hinged_boxes_scene()
    W = 10
    st = _hinged_states(sc, W, 6)
    ub = S.random_controls(sc.n_servos, W, seed=6, low=-2, high=2)
    g = np.random.default_rng(26).normal(size=st.shape)
    g[13 * sc.n_bodies:] = 0
    cfg = S.SolverConfig(budget=60, tol=1e-9, margin=0.5)        # the boxes are 0.2 m high: all 8 corners
    _compare(sc, cfg, ostrich, st, ub, H, "f64", 1e-7, 1e-6, 1e-6, 0.5, grads=g, threads=threads)


@pytest.mark.parametrize("dtype,per_sm", [("f32", 4), ("f64", 2)])
@pytest.mark.parametrize("kind,solver", [("robot", 0), ("box", 0), ("robot", 1)])
def test_results_do_not_depend_on_the_launch(ostrich, dtype, per_sm, kind, solver):  # noqa: F811
    """The first worlds of a launch one world larger than what runs with four warps each (two
    for the box, with normals and friction apart), against the same worlds alone."""
    sc = S.robot_box_scene() if kind == "robot" else S.box_drop_scene()
    W, n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 1, 6
    tdt = torch.float64 if dtype == "f64" else torch.float32
    if kind == "robot":
        st = S.robot_box_states(sc, n, seed=3)
    else:
        st = np.concatenate([S.box_drop_state(sc, 0.2 * k, -1e-3 * k) for k in range(n)], axis=1)
    st = np.repeat(st, -(-W // n), axis=1)[:, :W]
    st = st[:, np.argsort(np.arange(W) % n, kind="stable")]      # worlds of a kind side by side
    ub = S.random_controls(sc.n_servos, W, seed=3)
    g = np.random.default_rng(4).normal(size=st.shape)
    outs = []
    for cols in (np.arange(W), np.arange(0, W, W // n)[:n]):
        ctx = ostrich.Context(sc, S.SolverConfig(tol=1e-4, linear_solver=solver), len(cols), dtype=dtype, tape_slots=1)
        dev = [torch.tensor(np.ascontiguousarray(a[:, cols]), dtype=tdt, device="cuda") for a in (st, ub, g)]
        r = ctx.step(dev[0], dev[1], H, tape_slot=0)
        ds, du = ctx.adjoint(0, dev[2], H)
        torch.cuda.synchronize()
        outs.append([x.cpu() for x in (r["state"], r["impulses"], r["iters"].reshape(1, -1), ds, du)])
        ctx.close()
    pick = np.arange(0, W, W // n)[:n]
    for a, b in zip(*outs):
        assert torch.equal(a[:, pick], b)

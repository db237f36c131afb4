"""The adjoint of a world that holds a non-finite value.

A derivative of a product is formed as a' b + a b', so a non-finite factor makes it NaN
along every coordinate, the positions (whose own derivative is a unit vector) included.  A
gradient that came back finite in some entries there would be taken for one.

* a NaN velocity: the step returns a NaN iterate, and no entry of dL/dq- is finite;
* an infinite cotangent of one quaternion entry: that body's dL/dq- is not finite either;
* the other worlds of the launch: bit-identical to a launch without it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_08800_gb300 import scenes as S  # noqa: E402

H = 0.1
BAD = 1


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_08800_gb300 import ostrich
    ostrich.lib()
    return ostrich


def _states(kind):
    if kind == "robot":
        sc = S.robot_box_scene()
        return sc, S.robot_box_states(sc, 3, seed=14)
    sc = S.box_drop_scene()
    return sc, np.concatenate([S.box_drop_state(sc, 0.1 * k, -1e-3 if kind == "box" else 2.0) for k in range(3)], axis=1)


def _grads(M, sc, st, g, dtype, solver, exact):
    tdt = torch.float64 if dtype == "f64" else torch.float32
    W = st.shape[1]
    ctx = M.Context(sc, S.SolverConfig(tol=1e-4, linear_solver=solver), W, dtype=dtype, tape_slots=1)
    if exact:
        ctx.set_adjoint_mode(M.ADJ_EXACT)
    ub = S.random_controls(sc.n_servos, W, seed=3) if sc.n_servos else np.zeros((1, W))
    s_in, u_in, g_in = (torch.tensor(a, dtype=tdt, device="cuda") for a in (st, ub, g))
    ctx.step(s_in, u_in, H, tape_slot=0)
    ds, _ = ctx.adjoint(0, g_in, H)
    ds = ds.cpu()
    ctx.close()
    return ds


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("kind,solver,exact", [("free_box", 0, False), ("free_box", 0, True), ("free_box", 1, False),
                                               ("box", 0, False), ("box", 1, False), ("robot", 0, False),
                                               ("robot", 1, False)])
def test_nothing_finite_is_left_of_a_nan_world(M, kind, solver, exact, dtype):
    sc, st = _states(kind)
    nb = sc.n_bodies
    g = np.random.default_rng(7).normal(size=st.shape)
    g[13 * nb:] = 0
    bad = st.copy()
    bad[7 * nb + 1, BAD] = np.nan
    ds = _grads(M, sc, bad, g, dtype, solver, exact)
    ref = _grads(M, sc, st, g, dtype, solver, exact)
    assert torch.isnan(ds[:7 * nb, BAD]).all()
    assert torch.isfinite(ref).all()
    for w in (0, 2):
        assert torch.equal(ds[:, w], ref[:, w])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("kind", ["free_box", "box"])
def test_an_infinite_cotangent_reaches_every_position(M, kind, dtype):
    sc, st = _states(kind)
    g = np.random.default_rng(8).normal(size=st.shape)
    g[13:] = 0
    bad = g.copy()
    bad[4, BAD] = np.inf
    ds = _grads(M, sc, st, bad, dtype, 0, False)
    ref = _grads(M, sc, st, g, dtype, 0, False)
    assert not torch.isfinite(ds[:7, BAD]).any()
    for w in (0, 2):
        assert torch.equal(ds[:, w], ref[:, w])

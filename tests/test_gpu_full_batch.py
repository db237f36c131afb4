"""The kernel of large launches, for every thread count a context can be set to.

A launch of few worlds runs a kernel of its own, with at least 128 threads per world (64 for
scenes of at most 32 rows).  The parity tests hold a handful of worlds each, so it is that
kernel which they compare with the oracle.  Here the same worlds stand in a launch one world
larger than the line, which runs the other kernel with the context's 32, 64 or 128 threads,
and have to come out with the same bits: the step's state, impulses and iteration words, and
the adjoint.  Together the two carry the comparison over to every launch shape.

Scenes: groups of up to 16, 24 and 48 rows, separators of 0, 6, 24, 36 and 42 rows.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_08800_gb300 import scenes as S  # noqa: E402
from tests.test_gpu_parity import _hinged_states, ostrich  # noqa: E402,F401
from tests.test_gpu_shapes import vehicle_scene, vehicle_states  # noqa: E402
from tests.test_oracle_pins import hinged_boxes_scene  # noqa: E402

H = 0.1
N = 7


def _scene(kind):
    margin = 0.02
    if kind == "robot":
        sc = S.robot_box_scene()
        st = S.robot_box_states(sc, N, seed=5)
    elif kind == "box":
        sc = S.box_drop_scene()
        st = np.concatenate([S.box_drop_state(sc, 0.2 * k, -1e-3 * k) for k in range(N)], axis=1)
    elif kind == "terrain":
        sc = S.terrain_scene()
        st = S.terrain_states(sc, N, seed=5)
        st[2:7 * sc.n_bodies:7] -= 0.012                 # resting on the terrain
    elif kind == "hinged":
        sc = hinged_boxes_scene()
        st = _hinged_states(sc, N, 6)
        margin = 0.5                                     # all eight corners of a box
    else:
        sc, offs = vehicle_scene(int(kind[-1]))
        st = vehicle_states(sc, offs, N, 5)
    return sc, st, margin


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("threads", [32, 64, 128])
@pytest.mark.parametrize("kind", ["robot", "box", "terrain", "hinged", "vehicle6", "vehicle7"])
def test_large_launch_has_the_bits_of_a_small_one(ostrich, kind, threads, dtype):  # noqa: F811
    sc, st, margin = _scene(kind)
    few = (4 if dtype == "f32" else 2) * torch.cuda.get_device_properties(0).multi_processor_count
    tdt = torch.float64 if dtype == "f64" else torch.float32
    ub = S.random_controls(sc.n_servos, N, seed=5) if sc.n_servos else np.zeros((1, N))
    g = np.random.default_rng(6).normal(size=st.shape)
    outs = []
    for W in (few + 1, N):
        cols = np.arange(W) % N
        ctx = ostrich.Context(sc, S.SolverConfig(tol=1e-4, margin=margin), W, dtype=dtype, tape_slots=1, threads=threads)
        assert W == N or ctx.launch_threads() == threads
        dev = [torch.tensor(np.ascontiguousarray(a[:, cols]), dtype=tdt, device="cuda") for a in (st, ub, g)]
        r = ctx.step(dev[0], dev[1], H, tape_slot=0)
        ds, du = ctx.adjoint(0, dev[2], H)
        torch.cuda.synchronize()
        outs.append([x.cpu() for x in (r["state"], r["impulses"], r["ids"], r["iters"].reshape(1, -1), ds, du)])
        ctx.close()
    for big, small in zip(*outs):
        for w0 in range(0, few + 1, N):                  # every copy of the worlds
            n = min(N, few + 1 - w0)
            assert torch.equal(big[:, w0:w0 + n], small[:, :n])

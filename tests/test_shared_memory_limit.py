"""Scenes and settings at the edge of a CTA's 227 KB of shared memory (host only).

What a launch takes is the world's working set and the kernel's own variables: the scene in
working precision (3.4 KB in FP64) and the adjoint's lists.  A setting whose sum is beyond the
limit is refused when it is asked for, instead of failing at every launch."""
import ctypes

import pytest

from paper_2609_08800_gb300 import build as B
from paper_2609_08800_gb300 import ostrich as M
from paper_2609_08800_gb300 import scenes as S

OSTRICH_EINVAL = 1
LIMIT = 227 * 1024
STATIC = {0: 2432 + 496, 1: 3520 + 496}          # of the adjoint kernel (ptxas -v), FP32 and FP64
KRYLOV = 20


@pytest.fixture(scope="module")
def lib():
    B.build()
    return M.lib()


def _star(n_bodies, n_joints, n_servos, n_boxes, n_wheels):
    """Joints from body 0 to the next ones; boxes first, then wheels, then bodies without shape."""
    bodies = [S.Body(1.0, (1.0, 1.0, 1.0), S.SHAPE_BOX if i < n_boxes else
                     S.SHAPE_WHEEL if i < n_boxes + n_wheels else S.SHAPE_NONE, (0.1, 0.1, 0.1), 0.1, 0.05)
              for i in range(n_bodies)]
    joints = [S.Joint(0, j + 1, (0, 0, 0), (0, 0, 0), kp=50.0 if j < n_servos else 0.0) for j in range(n_joints)]
    return S.Scene("star", bodies, joints, S.Env(S.ENV_BOX), 0.5)


def _exact_bytes(lib, h, nb, dtype):
    """Dynamic shared memory of the exact adjoint: the working set, then the local Jacobians and
    the Krylov space, each array on an 8-byte boundary."""
    lay = (ctypes.c_int32 * 4)()
    lib.ostrich_layout(h, lay)
    m, ns = lay[1], max(lay[2], 1)
    n, sz, off = 6 * nb + m, 8 if dtype else 4, 0
    for c in (36 * nb * nb, 12 * m, 2 * ns, ns, (KRYLOV + 1) * n, (KRYLOV + 1) * KRYLOV, KRYLOV, KRYLOV, KRYLOV + 1,
              KRYLOV, n, n, n, 6 * nb, 4 * (KRYLOV + 2), 8):
        off = ((off + 7) & ~7) + sz * c
    return (lib.ostrich_workspace_bytes(h) + off + 15) & ~15


# scenes by the bytes their exact adjoint leaves of the limit: within the static variables (and
# so refused), beyond the limit by itself, and with room for them
@pytest.mark.parametrize("shape,left", [((8, 4, 1, 3, 5), "static"), ((8, 5, 3, 3, 4), "static"),
                                        ((8, 7, 1, 1, 5), "static"), ((7, 5, 4, 3, 4), "static"),
                                        ((8, 7, 7, 4, 4), "none"), ((8, 5, 2, 4, 3), "room"), ((5, 4, 4, 0, 4), "room")])
def test_exact_adjoint_counts_static_shared_memory(lib, shape, left):
    d, c, h = M.scene_desc(_star(*shape)), M.solver_cfg(S.SolverConfig()), ctypes.c_void_p()
    assert lib.ostrich_create(ctypes.byref(d), ctypes.byref(c), 4, 0, 1, 0, ctypes.byref(h)) == 0
    try:
        dyn = _exact_bytes(lib, h, shape[0], 1)
        assert left == ("none" if dyn > LIMIT else "static" if dyn + STATIC[1] > LIMIT else "room")
        rc = lib.ostrich_set_adjoint_mode(h, M.ADJ_EXACT, None)
        assert rc == (0 if left == "room" else OSTRICH_EINVAL)
        # the setting before stays in force, and is accepted again
        assert lib.ostrich_set_adjoint_mode(h, M.ADJ_PAPER, None) == 0
    finally:
        lib.ostrich_destroy(h)

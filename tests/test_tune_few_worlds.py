"""The autotuner on launches of few worlds, which run with more threads than the context's:
timing them says nothing about the candidates, so none is picked by noise and none recorded."""
import pytest

from paper_2609_08800_gb300 import tune

torch = pytest.importorskip("torch")


class _Ctx:
    """A context whose launches run with at least `floor` threads per world."""
    dtype, m_max, n_worlds = torch.float32, 120, 8

    def __init__(self, floor, threads=64):
        self.floor, self.threads, self.schedule = floor, threads, 0

    def set_threads(self, t):
        self.threads = t

    def set_schedule(self, s):
        self.schedule = s

    def launch_threads(self, n=None):
        return max(self.threads, self.floor)


def _tune(monkeypatch, tmp_path, ctx, ms):
    monkeypatch.setattr(tune, "key", lambda c, device=None: "f32:m128:dev")
    monkeypatch.setattr(tune, "time_step", lambda c, *a, **k: ms[c.threads] + c.schedule)
    path = tmp_path / "table.json"
    return tune.tune(ctx, None, None, 0.1, path=path), tune._load(path)


@pytest.mark.parametrize("floor,own,fastest,best", [(128, 64, 32, 64), (128, 32, 128, 32), (64, 64, 32, 64),
                                                    (64, 64, 128, 128)])
def test_few_worlds_keep_the_setting_and_record_nothing(monkeypatch, tmp_path, floor, own, fastest, best):
    ctx = _Ctx(floor, own)
    (t, times), table = _tune(monkeypatch, tmp_path, ctx, {c: 1.0 if c == fastest else 1.01 for c in tune.CANDIDATES})
    assert t == best == ctx.threads and set(times) == set(tune.CANDIDATES)
    assert table == {}


@pytest.mark.parametrize("fastest", tune.CANDIDATES)
def test_a_full_batch_records_the_fastest(monkeypatch, tmp_path, fastest):
    ctx = _Ctx(0)
    (t, times), table = _tune(monkeypatch, tmp_path, ctx, {c: 1.0 if c == fastest else 1.01 for c in tune.CANDIDATES})
    assert t == fastest == ctx.threads and ctx.schedule == 0
    assert table["f32:m128:dev"]["threads"] == fastest


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,per_sm", [("f32", 4), ("f64", 2)])
@pytest.mark.parametrize("kind,solver,few", [("robot", 0, 128), ("box", 0, 64), ("robot", 1, 32)])
def test_threads_of_a_launch(dtype, per_sm, kind, solver, few):
    """The library's answer on both sides of the line between few worlds and many."""
    from paper_2609_08800_gb300 import scenes as S
    from paper_2609_08800_gb300.ostrich import Context
    sc = S.robot_box_scene() if kind == "robot" else S.box_drop_scene()
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    ctx = Context(sc, S.SolverConfig(linear_solver=solver), 8, dtype=dtype, tape_slots=0)
    for t in tune.CANDIDATES:
        ctx.set_threads(t)
        assert ctx.launch_threads() == ctx.launch_threads(n) == max(t, few)
        assert ctx.launch_threads(n + 1) == t
    assert ctx.launch_threads(0) == 0
    ctx.close()

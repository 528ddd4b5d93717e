"""The tuners leave the choice of path with the library where it had it (CPU: a stand-in network whose
step time depends on the path and schedule in force)."""
import pytest

from paper_2410_13055_gb300 import autotune


class _Event:
    clock = [0.0]

    def __init__(self, enable_timing=True):
        self.t = None

    def record(self):
        self.t = _Event.clock[0]

    def elapsed_time(self, end):
        return end.t - self.t


class _Net:
    def __init__(self, auto, auto_ms):
        import torch
        self.auto, self.auto_ms = auto, auto_ms
        self.sched = {"bus_staged": 0, "bat_warps": 2}
        self.s = torch.zeros(4)

    def schedule(self):
        return dict(self.sched)

    def set_schedule(self, **kw):
        self.sched, self.auto = dict(kw), False

    def use_persistent(self, on):
        self.auto = False

    def set_opts(self, **kw):
        pass

    def auto_path(self):
        self.auto = True

    def path_is_auto(self):
        return self.auto

    def state(self, adjoint=False):
        return self.s

    def step(self, eta):
        _Event.clock[0] += self.auto_ms if self.auto else 10.0 + self.sched["bus_staged"] + self.sched["bat_warps"]


@pytest.mark.parametrize("auto,auto_ms,after", [(True, 5.0, True), (True, 11.1, True), (True, 30.0, False),
                                                (False, 5.0, False)])
def test_step_tuner_and_the_librarys_choice(monkeypatch, auto, auto_ms, after):
    import torch
    monkeypatch.setattr(torch.cuda, "Event", _Event)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a, **k: None)
    net = _Net(auto, auto_ms)
    out = autotune.tune_schedule_step(net, torch.zeros(2), step=net.step, steps=1, reps=1, margin=0.02)
    assert len(out["trials"]) == 6 and out["best"] == net.schedule()
    assert net.auto is after
    assert ("auto" in out) == auto
    if auto:
        assert out["auto"]["kept"] is after and out["auto"]["ms_per_step"] == pytest.approx(auto_ms)


def test_setting_with_no_path_gives_the_choice_back():
    net = _Net(True, 1.0)
    autotune._apply(net, {"persistent": None, "bus_staged": 1, "bat_warps": 2, "rho": 0.2})
    assert net.auto and net.schedule() == {"bus_staged": 1, "bat_warps": 2}
    autotune._apply(net, {"persistent": False, "bus_staged": 1, "bat_warps": 2})
    assert not net.auto

"""Autotuner logic on the CPU, against a simulation and events that keep a
clock of their own."""
import pytest

from paper_2212_14153_gb300 import autotune, fpd
from paper_2212_14153_gb300 import workloads as wl

CHUNK, BUFFERS, CAPTURE = 32, 4, 5.0  # steps a graph, graphs by step count, ms a capture


class Clock:
    now = 0.0


class FakeSimulation:
    """Captures step graphs as fpd_step and fpd_prepare do: by the step count
    modulo the mask buffers, dropped when the variant changes."""
    cost = [0.010, 0.011, 0.012, 0.013, 0.014]  # ms a step
    failing = None
    made = 0

    def __init__(self, cfg, stream=None, **kw):
        type(self).made += 1
        self.t, self.v, self.graphs = 0, 0, set()

    def tuning(self):
        return self.v, len(self.cost)

    def set_tuning(self, v):
        if v != self.v:
            self.v, self.graphs = v, set()

    def _plan(self, n):
        t = self.t
        while n:
            k = CHUNK if t >= 1 and n >= CHUNK else 1
            yield t % BUFFERS, k
            t, n = t + k, n - k

    def _capture(self, p):
        if p not in self.graphs:
            self.graphs.add(p)
            Clock.now += CAPTURE

    def prepare(self, n):
        for p, k in self._plan(n):
            if k > 1:
                self._capture(p)

    def step(self, n):
        for p, k in list(self._plan(n)):
            if k > 1:
                self._capture(p)
            Clock.now += k * self.cost[self.v]
            self.t += k

    def sync(self):
        if self.v == self.failing:
            raise fpd.FpdError(fpd.FPD_ETIMEOUT, "a bulk copy did not arrive")

    def close(self):
        pass


class FakeEvent:
    def __init__(self, enable_timing=False):
        pass

    def record(self, stream):
        self.at = Clock.now

    def synchronize(self):
        pass

    def elapsed_time(self, other):
        return other.at - self.at


class FakeStream:
    cuda_stream = 0


@pytest.fixture
def fakes(monkeypatch, tmp_path):
    import torch
    monkeypatch.setenv("FPD_TUNING_CACHE", str(tmp_path / "tuning.json"))
    monkeypatch.setattr(fpd, "Simulation", FakeSimulation)
    monkeypatch.setattr(torch.cuda, "Event", FakeEvent)
    monkeypatch.setattr(torch.cuda, "Stream", FakeStream)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "GPU")
    monkeypatch.setattr(FakeSimulation, "failing", None)
    monkeypatch.setattr(FakeSimulation, "made", 0)


CFG = wl.couette_only(40, 24, precision=1)


@pytest.mark.parametrize("steps,warmup", [(256, 64), (128, 32), (32, 0), (1, 7)])
def test_no_graph_is_captured_within_a_timing(fakes, steps, warmup):
    ms = autotune.time_variants(CFG, steps=steps, warmup=warmup)
    assert ms == pytest.approx(FakeSimulation.cost, rel=1e-9)


def test_a_variant_whose_run_fails_is_not_timed_in_silence(fakes, monkeypatch):
    monkeypatch.setattr(FakeSimulation, "failing", 3)
    with pytest.raises(fpd.FpdError):
        autotune.time_variants(CFG)


def test_constant_rates_are_not_timed(fakes):
    # every variant runs the same kernel there: their timings differ by noise
    assert autotune.tune(dict(CFG, collision=fpd.FPD_MRT_LL)) == 0
    assert FakeSimulation.made == 0
    assert autotune.tune(dict(CFG, collision=fpd.FPD_BGK)) == 0 and FakeSimulation.made == 1


@pytest.mark.parametrize("change", [dict(collision=2), dict(periodic_y=1), dict(gx=1e-5), dict(gy=-1e-5),
                                    dict(sandwich_zl=8.0, sandwich_zr=16.0), dict(a=3.0), dict(xi=0.5),
                                    dict(phi_cut=6.0), dict(n_beads=4, n_fibers=3), dict(n_beads=3), dict(nx=97),
                                    dict(precision=0)])
def test_the_cache_tells_workloads_of_other_kernels_apart(fakes, change):
    import numpy as np
    cfg = wl.random_fiber(np.random.default_rng(1), 96, 48, n_beads=6, a=2.0, xi=1.0, n_fibers=2, precision=1)
    autotune.tune(cfg)
    autotune.tune(dict(cfg, u_top=0.011, theta0=[0.1, 0.2]))  # the same kernels on the same work
    assert FakeSimulation.made == 1
    autotune.tune(dict(cfg, **change))
    assert FakeSimulation.made == 2

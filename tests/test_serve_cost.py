"""The tile costs by which shared launches split their CTAs (serve.Server._time_impl): timed
on the launch that the shared mode runs, not on a pack's own (two CTAs an SM at orders 2
and 3).  On the CPU, with a clock that each kind of launch advances by its own amount."""
from types import SimpleNamespace

import pytest

from paper_0901_1024_gb300 import Mesh, serve

OWN_MS, SHARED_MS, SMS = 0.120, 0.176, 152     # a stage of a pack alone, and in a shared launch


class Clock:
    now = 0.0


class Event:
    def __init__(self, enable_timing):
        assert enable_timing

    def record(self, stream):
        self.t = Clock.now

    def synchronize(self):
        pass

    def elapsed_time(self, other):
        return other.t - self.t


class Pack:
    def __init__(self, torch, N, solves, old, padding, impl, graphs, stream, shape=0):
        self.N, self.K, self.parity, self.mesh = N, sum(s.K for s in solves), 0, object()
        self.res = self.dt_elem = None

    def buffers(self):
        return None, None

    def step(self):
        Clock.now += 5 * OWN_MS
        self.parity ^= 1

    def release(self):
        pass


@pytest.mark.parametrize("N,K,expected_ms", [(1, 4000, SHARED_MS), (2, 20000, SHARED_MS),
                                             (3, 700, SHARED_MS), (6, 4000, SHARED_MS),
                                             (7, 4000, OWN_MS)])
def test_cost_of_a_tile_in_a_shared_launch(monkeypatch, N, K, expected_ms):
    def shared(meshes, src, dst, res, stage, dt=1.0, dt_elem=None, tile_cost=None, stream=None):
        assert len(meshes) == 1
        Clock.now += SHARED_MS
    monkeypatch.setattr(serve, "_Pack", Pack)
    monkeypatch.setattr(serve.Mesh, "rk_stage_multi", staticmethod(shared))
    monkeypatch.setattr(serve.Server, "_cost", {})
    monkeypatch.setattr(serve.Server, "_pad_mesh", lambda self, N: None)
    cuda = SimpleNamespace(Event=Event, current_device=lambda: 0, get_device_properties=lambda d:
                           SimpleNamespace(multi_processor_count=SMS))
    srv = serve.Server.__new__(serve.Server)
    srv.torch, srv.stream, srv.stats = SimpleNamespace(cuda=cuda), None, {}
    solves = [SimpleNamespace(K=K, bytes=1.0)]
    ms = srv._time_impl(N, solves, Mesh.STAGE_TC)
    assert ms == pytest.approx(15 * OWN_MS)            # the choice of kernel: the pack's own launch
    tiles = -(-K // (20 if N <= 4 else 8))
    assert srv._cost[srv._tune_key(N, solves)] == pytest.approx(
        expected_ms * min(tiles, SMS) / tiles)
    assert srv.stats["model_now"] == 0

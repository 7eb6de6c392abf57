"""The slice products' schedule in a process group of several ranks: no candidate
shares tiles between CTAs by TMA multicast (no GPU needed)."""
import pytest

from paper_1911_11906_gb300 import autotune as A

torch = pytest.importorskip("torch")


class Recorder:
    def lookup(self, name, fields, candidates):
        self.candidates = list(candidates)
        return self.candidates[-1]


@pytest.mark.parametrize("world,clusters", [(1, {"1", "2"}), (2, {"1"}), (8, {"1"})])
def test_clusters_of_a_process_group(monkeypatch, world, clusters):
    monkeypatch.setattr(A, "_device_name", lambda: "none")
    monkeypatch.setattr(torch.distributed, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.distributed, "get_world_size", lambda *a: world)
    tuner = Recorder()
    sched = A.best_ozaki_schedule(640, tuner=tuner)
    assert {c.split("/")[3] for c in tuner.candidates} == clusters
    assert str(sched["ozaki_cluster"]) in clusters

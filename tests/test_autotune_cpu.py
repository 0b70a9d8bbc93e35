"""The autotuner's search, on a driver that only records what is tried."""
from types import SimpleNamespace

import pytest

from paper_2604_16613_gb300 import autotune as A


class Recorder:
    def __init__(self, max_qubits):
        self.bounds = SimpleNamespace(max_qubits=max_qubits)
        self.tuning = dict(stage1_threads=512, stage1_blocks_per_sm=0, stage2_threads=512, stage2_blocks_per_sm=8,
                           obs_words=4, obs_segments=3, stage1_wide_emit=0)
        self.tried = []

    def get_tuning(self):
        return dict(self.tuning)

    def set_tuning(self, **t):
        self.tuning = dict(t)


@pytest.mark.parametrize("max_qubits", [31, 32, 480, 481, 2520, 2521])
def test_no_trial_differs_in_what_changes_no_launch(max_qubits, monkeypatch):
    split = max_qubits < 32 or 480 < max_qubits <= 2520

    def fake_time(driver, circuits, noise, level, repeats):
        driver.tried.append(dict(driver.tuning))
        return 1.0 - 1e-3 * len(driver.tried)          # every later trial looks a little faster: noise
    monkeypatch.setattr(A, "_time", fake_time)
    monkeypatch.setattr(A, "_cache", {})
    drv = Recorder(max_qubits)
    circuit = SimpleNamespace(n_qubits=max_qubits, n_ops=1, n_observables=12)
    best = A.autotune(drv, circuit, None)
    threads, segments = {t["stage1_threads"] for t in drv.tried}, {t["obs_segments"] for t in drv.tried}
    if split:
        assert threads == {256, 512, 1024} and segments == {1, 2, 3}
    else:
        assert threads == {512} and segments == {3}
        assert best["stage1_threads"] == 512 and best["obs_segments"] == 3
    assert {t["stage1_blocks_per_sm"] for t in drv.tried} == {0, 1}
    assert {t["obs_words"] for t in drv.tried} == {1, 2, 4, 8}

"""The tuner keeps a setting that nothing beats by more than repeated timings differ."""
from __future__ import annotations

from paper_2508_20403_gb300 import autotune as AT


def test_noise_changes_no_setting():
    times = iter([1.0, 0.995, 1.004, 0.991, 0.999, 0.9901, 1.01, 0.993])
    best, t, tried = AT.coordinate_descent(lambda s: next(times))
    assert best == {k: v[0] for k, v in AT.SPACE.items()} and t == 1.0 and len(tried) == 8


def test_gains_do():
    space = {"a": [0, 1], "b": [0, 1]}
    best, t, _ = AT.coordinate_descent(lambda s: 1.0 - 0.02 * s["a"] + 0.5 * s["b"], space)
    assert best == {"a": 1, "b": 0} and t == 0.98

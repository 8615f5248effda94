"""The benchmark's byte model follows the launch plan that runs."""
import json

import pytest

import bench


def compact(n):
    return 3 * (2 * (n // 3) + 1) ** 2 * 8


def mixed(n, N):
    return 3 * (2 * (n // 3) + 1) * N * 8


@pytest.mark.parametrize("n,plan,want", [
    (128, (4, 0), 14 * compact(128)),                                    # persistent step: 14 compact passes
    (256, (6, 3), 14 * compact(256)),                                    # whatever the row variant
    (160, (0, 0), 14 * compact(160)),                                    # no power of two: its one plan
    (128, (1, 9), 16 * mixed(128, 128) + 14 * compact(128)),             # two kernels on n points
    (512, (5, 9), 16 * mixed(512, 384) + 12 * compact(512)),             # 3n/4 points, as a pair only
    (512, (5, 8), 16 * mixed(512, 512) + 14 * compact(512)),
    (512, (6, 9), 16 * mixed(512, 512) + 14 * compact(512)),
    (1024, (6, 7), 16 * mixed(1024, 768) + 12 * compact(1024)),
    (1024, (5, 7), 16 * mixed(1024, 1024) + 14 * compact(1024)),
])
def test_step_bytes(n, plan, want):
    assert bench.step_bytes_of(n, 1, plan) == want
    assert bench.step_bytes_of(n, 7, list(plan)) == 7 * want


def test_traffic_is_of_a_pair():
    assert set(bench.FINE_TRAFFIC) == {("fine row kernel", (6, 7)), ("fine column kernel", (6, 7))}


def test_tuned_plan(tmp_path):
    f = tmp_path / "tune.json"
    entry = {"device": "G", "n": 64, "prec": 0, "batch": 32, "col": 4, "row": 0, "ms_per_step": 0.1}
    f.write_text(json.dumps({"kd_autotune": 1, "entries": [dict(entry, prec=1, col=9), dict(entry, n=128, col=8), entry]}))
    assert bench.tuned_plan(str(f), "G", 64, 32) == bench.tuned_plan(str(f), "G", 64, 17) == (4, 0)
    with pytest.raises(RuntimeError):
        bench.tuned_plan(str(f), "G", 64, 33)

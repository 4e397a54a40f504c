"""The bench's roofline entry of a pass of four steps, from the timed region."""
import os
import sys
import types

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_pass_roofline():
    import bench
    w = types.SimpleNamespace(nodes=1_000_000, name="w")
    # 40 steps in 10 passes of three launches; 0.2 ms a pass
    r = bench.pass_roofline(w, "f32dev", 2.0, 40, 30, 6800.0)
    assert r["avg_launch_us"] == 200.0 and r["algorithmic_bytes_per_launch"] == 72_000_000
    assert r["achieved"] == pytest.approx(360.0) and r["frac"] == pytest.approx(360.0 / 6800.0, abs=1e-4)
    # single steps launch two kernels each; fewer steps than a pass
    assert bench.pass_roofline(w, "f32dev", 2.0, 40, 80, 6800.0) is None
    assert bench.pass_roofline(w, "f32dev", 2.0, 3, 2, 6800.0) is None

"""The step number in an EUNSTABLE report: the first step with rho <= 0 or NaN is
the same whether that step is taken alone, inside a pass of four, or among the
single steps after one, whose link kernel may still be running."""
import re

import numpy as np
import pytest

from paper_2210_10377_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_10377_gb300 import binding
    binding.lib()
    return binding


def reported(gb, lat, n):
    with pytest.raises(gb.LbmError) as e:
        lat.step(n)
    assert e.value.code == 4
    return int(re.search(r"step (\d+)", str(e.value)).group(1))


@pytest.mark.parametrize("storage", ["f64", "f32dev", "f16dev"])
def test_first_unstable_step_does_not_depend_on_the_split(gb, storage):
    nx, ny = 200, 64
    m = np.zeros((ny, nx), np.uint8)
    m[20:44:2, 40:60] = 1  # many links
    f0 = inputs.random_populations(nx, ny, seed=8, lo=0.08, hi=0.14)

    def fresh():
        lat = gb.Lattice(m, 0.5001, 0.1, storage=storage)
        lat.set_populations(f0)
        return lat

    lat = fresh()
    for first in range(400):
        try:
            lat.step(1)
        except gb.LbmError as e:
            assert "step %d" % first in str(e)
            break
    lat.close()
    assert 12 < first < 399
    for k in range(1, 5):  # k single steps, then passes: step `first` falls in a pass or in its rest
        lat = fresh()
        for _ in range(k):
            lat.step(1)
        assert reported(gb, lat, first - k + 1) == first
        lat.close()
        lat = fresh()
        for _ in range(k):
            lat.step(1)
        assert reported(gb, lat, 2 * first) == first
        lat.close()


@pytest.mark.parametrize("storage", ["f32", "f16dev"])
def test_a_report_is_given_once_and_the_next_one_is_its_own(gb, storage):
    # the status words are cleared after a report, and only then
    nx, ny = 200, 64
    lat = gb.Lattice(np.zeros((ny, nx), np.uint8), 0.5001, 0.1, storage=storage)
    calm = lat.populations()
    wild = inputs.random_populations(nx, ny, seed=8, lo=0.08, hi=0.14)
    reports = []
    for _ in range(2):
        lat.set_populations(wild)
        t0 = lat.steps_done
        reports.append(reported(gb, lat, 399) - t0)
        lat.set_populations(calm)
        for n in (1, 9, 1):
            lat.step(n)
    assert reports[0] == reports[1]
    lat.close()

"""Device memory of the passes of four steps: taken by the handles that run them
and no others, and done without where the allocator refuses it."""
import numpy as np
import pytest

from paper_2210_10377_gb300 import inputs

pytestmark = pytest.mark.gpu

NX, NY = 300, 64
STATE = {"f64": 8, "f32": 4, "f32dev": 4, "f16dev": 2}


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_10377_gb300 import binding
    binding.lib()
    return binding


def lattice(gb, storage, **kw):
    m = np.zeros((NY, NX), np.uint8)
    m[28:36, 90:110] = 1
    return gb.Lattice(m, 0.6, inputs.random_inlet(NY, seed=7), storage=storage, **kw)


def held(lat):
    return sum(lat._alloc.live.values())


def state(storage):
    return 9 * NY * 320 * STATE[storage]  # rows of 300 nodes are 320 apart


@pytest.mark.parametrize("storage", ["f64", "f32dev", "f16dev"])
def test_only_steps_taken_in_passes_take_their_memory(gb, storage):
    for kw in (dict(kernel="staged"), dict()):
        lat = lattice(gb, storage, **kw)
        before = held(lat)
        lat.step(1)
        if kw:
            lat.prepare(100)
            lat.step(40)  # the staged kernel
        else:
            lat.set_kernel_timing(True)
            lat.step(20)  # one launch at a time
            lat.set_kernel_timing(False)
            lat.step(3)
        assert held(lat) == before, kw
        lat.close()


@pytest.mark.parametrize("storage", ["f64", "f32dev"])
def test_kept_steps_of_a_gradient_take_no_states_of_passes(gb, storage):
    lat = lattice(gb, storage)
    before = held(lat)
    lat.adjoint(12, 5, 0.3, 0.7)
    assert held(lat) - before < state(storage)
    lat.close()

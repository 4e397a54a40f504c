"""lbm_adjoint from a state that steps have already left post-collision: the
kept forward steps then start with a group of four at once, also when there
are just four of them.  Each plan (states kept, every state checkpointed)
gives the same bits."""
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


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("steps", [3, 4, 5, 8, 9])
def test_kept_steps_from_a_post_collision_state(gb, storage, steps):
    ny, nx = 40, 150
    m = np.zeros((ny, nx), np.uint8)
    m[15:24, 50:62] = 1
    u = inputs.random_inlet(ny, seed=7)
    runs = []
    for K in (0, 1):  # keep every state; checkpoint every state
        lat = gb.Lattice(m, 0.6, u, storage=storage)
        lat.step(1)
        outs = [lat.adjoint(steps, steps, 0.4, 0.9, checkpoint_every=K) for _ in range(2)]
        outs.append((lat.populations(), *lat.force_series("B"), *lat.force_series("DRTT")))
        runs.append(outs)
        lat.close()
    for kept, checked in zip(*runs):
        for a, b in zip(kept, checked):
            assert np.array_equal(a, b)

"""The bounded waits of the multi-step kernel, without any GPU fault: with the
poll bound at zero every CTA's first wait for its staged rows gives up, the CTA
lets its copies land and leaves, lbm_step reports ETIMEOUT, and the handle,
given a state back, steps on like a fresh one."""
import numpy as np
import pytest

from paper_2210_10377_gb300 import inputs

pytestmark = pytest.mark.gpu

ETIMEOUT = 5


@pytest.fixture(scope="module")
def gb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2210_10377_gb300 import binding
    binding.lib()
    return binding


# a partial strip alone; strips with the inlet, the outlet and a body; FP32
# takes the multi-step kernel from 600,000 nodes on
@pytest.mark.parametrize("storage,nx,ny", [("f16dev", 64, 17), ("f16dev", 500, 131), ("f32dev", 1201, 501)])
def test_an_expired_wait_is_reported_and_the_handle_recovers(gb, storage, nx, ny):
    m = np.zeros((ny, nx), np.uint8)
    m[ny // 2, nx // 3:nx // 3 + 3] = 1
    u = inputs.random_inlet(ny, seed=3, amp=0.002)
    lat = gb.Lattice(m, 0.56, u, storage=storage)
    lat.step(33)
    f = lat.populations()
    lat.set_wait_limit(0)
    lat.step(3)  # single steps of the direct kernel wait on nothing
    with pytest.raises(gb.LbmError) as e:
        lat.step(8)
    assert e.value.code == ETIMEOUT
    with pytest.raises(gb.LbmError) as e:
        lat.step(60)  # again, from captured graphs
    assert e.value.code == ETIMEOUT
    lat.set_wait_limit(-1)
    lat.set_populations(f)
    t0 = lat.steps_done
    lat.step(62)
    ref = gb.Lattice(m, 0.56, u, storage=storage)
    ref.set_populations(f)
    ref.step(62)
    assert np.array_equal(lat.populations(), ref.populations())
    for s in ("A", "B", "A_RTT", "SI"):
        assert np.array_equal(np.stack(lat.force_series(s, t0, 62)), np.stack(ref.force_series(s, 0, 62))), s
    ref.close()
    lat.close()

"""Steps taken in passes of four, by graphs long and short, behind one another
and beside single steps, against the same steps taken one call at a time: the
same bits in the populations and in every force series, with and without a body
force, in channels and periodic domains."""
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


def block(nx, ny):
    m = np.zeros((ny, nx), np.uint8)
    m[ny // 2 - 4:ny // 2 + 4, nx // 3:nx // 3 + 12] = 1
    return m


# calls of two and three steps from rest and behind passes; the short and the
# long graphs, opened by a held link kernel and not; a rest of every length
CHUNKS = [1, 3, 2, 13, 63, 3, 50, 400, 2, 110]


def compare(gb, m, storage, chunks, **kw):
    ny, nx = m.shape
    u = inputs.random_inlet(ny, seed=3, amp=0.002)
    runs = []
    for calls in (chunks, [1] * sum(chunks)):
        lat = gb.Lattice(m, 0.56, u, storage=storage, **kw)
        lat.set_populations(lat.populations() * inputs.perturbation(nx, ny, seed=4))
        for n in calls:
            lat.step(n)
        runs.append([lat.populations()] + [np.stack(lat.force_series(s)) for s in ("A", "B", "A_RTT", "SI", "DRTT")])
        lat.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f64", "f32", "f32dev", "f16dev"])
def test_every_graph_and_rest(gb, storage):
    compare(gb, block(260, 50), storage, CHUNKS)


@pytest.mark.parametrize("storage,nx,ny", [("f64", 150, 40), ("f32", 257, 66), ("f32dev", 257, 66), ("f16dev", 241, 96),
                                           ("f32", 1201, 501), ("f32dev", 1300, 467)])
def test_channel_with_a_body_force(gb, storage, nx, ny):
    compare(gb, block(nx, ny), storage, [1, 4, 3, 14, 9], body_force=(2e-6, -1e-6))


@pytest.mark.parametrize("storage,nx,ny", [("f64", 150, 41), ("f32", 261, 66), ("f32dev", 130, 35), ("f16dev", 241, 96),
                                           ("f16dev", 128, 48)])
@pytest.mark.parametrize("whole", [False, True])
def test_periodic_domain(gb, storage, nx, ny, whole):
    # bodies across both edges; the box inside the domain and all of it
    m = block(nx, ny)
    m[:3, 30:36] = m[-2:, 30:36] = 1
    m[10:14, :2] = m[10:14, -3:] = 1
    kw = dict(cv=[0, nx - 1, 0, ny - 1]) if whole else {}
    compare(gb, m, storage, [1, 4, 3, 14, 25], kind=gb.PERIODIC, body_force=(2e-6, -1e-6), **kw)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
def test_batch_every_graph_and_rest(gb, storage):
    domains = [dict(mask=block(nx, ny), tau=t, u_in=inputs.random_inlet(ny, seed=ny, amp=0.002))
               for nx, ny, t in ((150, 40, 0.6), (260, 50, 0.56), (64, 33, 0.8))]
    chunks = [1, 3, 2, 13, 50, 3, 110, 2, 70]
    runs = []
    for calls in (chunks, [1] * sum(chunks)):
        b = gb.Batch(domains, storage=storage)
        for n in calls:
            b.step(n)
        runs.append([x for d in range(3) for x in (b.populations(d), *b.force_series(d, "A"), *b.force_series(d, "B"),
                                                   *b.force_series(d, "SI"), *b.force_series(d, "DRTT"))])
        b.close()
    for x, y in zip(*runs):
        assert np.array_equal(x, y)

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


@pytest.fixture
def refusing(gb, monkeypatch):
    """An allocator whose user can set the largest block that it hands out."""
    limit = [None]
    alloc = gb._TorchAllocator._alloc

    def limited(self, nbytes, stream, user):
        return None if limit[0] is not None and nbytes > limit[0] else alloc(self, nbytes, stream, user)

    monkeypatch.setattr(gb._TorchAllocator, "_alloc", limited)
    return limit


@pytest.mark.parametrize("storage", ["f64", "f16dev"])
def test_populations_need_room_for_one_plane_only(gb, refusing, storage):
    lat = lattice(gb, storage)
    lat.step(5)
    want = lat.populations()
    refusing[0] = 8 * NX * NY + 255  # one FP64 plane, rounded up to 256 bytes
    assert np.array_equal(lat.populations(), want)
    refusing[0] = 8 * NX * NY - 1
    with pytest.raises(gb.LbmError) as e:
        lat.populations()
    assert e.value.code == 2
    lat.close()


@pytest.mark.parametrize("storage", ["f64", "f32dev", "f16dev"])
def test_without_room_for_passes_steps_run_one_by_one(gb, refusing, storage):
    runs = []
    for refuse in (False, True):
        refusing[0] = None
        lat = lattice(gb, storage)
        if refuse:
            before = held(lat)
            refusing[0] = 1024  # neither the states nor the rows of the passes
        for n in (1, 30, 7):
            lat.step(n)
        if refuse:
            assert held(lat) == before
        refusing[0] = None
        runs.append((lat.populations(), np.stack(lat.force_series("B")), np.stack(lat.force_series("DRTT"))))
        lat.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


def test_a_batch_without_room_for_passes_gives_back_what_it_got(gb, refusing):
    m = np.zeros((NY, NX), np.uint8)
    m[28:36, 90:110] = 1
    domains = [dict(mask=m, tau=0.6, u_in=0.05), dict(mask=np.zeros((40, 100), np.uint8), tau=0.7, u_in=0.03)]
    runs = []
    for refuse in (False, True):
        refusing[0] = None
        b = gb.Batch(domains, storage="f32")
        if refuse:
            before = held(b)
            refusing[0] = state("f32")  # the tables of the passes, not their states
        for n in (1, 30, 7):
            b.step(n)
        if refuse:
            assert held(b) == before
        refusing[0] = None
        runs.append([b.populations(0), b.populations(1), *b.force_series(0, "B"), *b.force_series(0, "DRTT")])
        b.close()
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


def test_preparing_fewer_steps_than_a_pass_takes_no_memory_for_passes(gb):
    for storage in ("f64", "f16dev"):
        lat = lattice(gb, storage)
        before = held(lat)
        lat.prepare(3)
        assert held(lat) == before
        lat.prepare(4)
        taken = held(lat)
        assert taken > before
        lat.step(4)
        lat.step(4)
        assert held(lat) == taken
        lat.close()
    b = gb.Batch([dict(mask=np.zeros((40, 100), np.uint8), tau=0.7, u_in=0.03)], storage="f32")
    before = held(b)
    b.prepare(3)
    assert held(b) == before
    b.prepare(4)
    assert held(b) > before
    b.close()


@pytest.mark.parametrize("torch_alloc", [True, False])
@pytest.mark.parametrize("storage", ["f64", "f32dev", "f16dev"])
def test_calls_before_the_passes_are_set_up(gb, storage, torch_alloc):
    # short calls run one by one until enough steps were asked for; the same bits
    runs = []
    for chunks in ([5, 3, 7, 4, 9, 12, 30, 2], [1] * 72):
        lat = lattice(gb, storage, torch_alloc=torch_alloc)
        for n in chunks:
            lat.step(n)
        runs.append([lat.populations()] + [np.stack(lat.force_series(s)) for s in ("A", "B", "SI", "DRTT")])
        lat.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)

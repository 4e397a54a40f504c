"""Passes of four steps (lbm_march.cu; on small grids single-step launches with
one link kernel) against single steps: the staged kernel takes single steps on
any grid, the direct kernel four at a time where the grid takes passes.  The populations and the link sums are the same bits, the
box sums too up to the order in which the staged kernel adds them."""
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


def body(name, nx, ny):
    """none; a disc inside; one at the inlet, one at the outlet; one that wraps through the top."""
    m = np.zeros((ny, nx), np.uint8)
    if name == "none":
        return m
    r = max(1.0, min(nx, ny) / 14)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    cx, cy = {"disc": (0.4 * nx, 0.5 * ny), "inlet": (2 + r, 0.55 * ny), "outlet": (nx - 3 - r, 0.45 * ny), "wrap": (0.3 * nx, 0.0)}[name]
    dy = np.abs(y - cy)
    m[(x - cx) ** 2 + np.minimum(dy, ny - dy) ** 2 <= r * r] = 1
    m[:, :2] = 0
    m[:, nx - 2:] = 0
    return m


# strips of 120 columns (16: one partial strip; 121 and 241: the outlet column
# alone in the last one; 119 .. 123: the outlet in the halo of the strip
# before), odd columns and rows, pieces of an odd number of rows; FP32 grids
# take passes of the multi-step kernel from 600,000 nodes on
SIZES = [("f16dev", nx, ny) for nx, ny in
         [(16, 16), (64, 17), (119, 16), (120, 33), (121, 40), (122, 41), (123, 64), (240, 51), (241, 96), (500, 255)]]
SIZES += [("f32dev", 1201, 751), ("f32", 1200, 751), ("f32dev", 1319, 700)]
# small grids of the other storages: passes of single-step launches
SIZES += [("f64", 131, 35), ("f32dev", 257, 66)]


@pytest.mark.parametrize("storage,nx,ny", SIZES)
@pytest.mark.parametrize("name", ["none", "disc", "inlet", "outlet", "wrap"])
def test_passes_equal_single_steps(gb, storage, nx, ny, name):
    m = body(name, nx, ny)
    u = inputs.random_inlet(ny, seed=3, amp=0.002)
    start = None
    runs = []
    for kernel, chunks in (("staged", [30]), ("direct", [1, 4, 3, 8, 14])):
        lat = gb.Lattice(m, 0.56, u, storage=storage, kernel=kernel)
        if start is None:
            start = lat.populations() * inputs.perturbation(nx, ny, seed=4)
        lat.set_populations(start)
        for n in chunks:
            lat.step(n)
        runs.append((lat.populations(), {s: np.stack(lat.force_series(s)) for s in ("A", "B", "A_RTT", "SI", "DRTT")}))
        lat.close()
    (f_ref, s_ref), (f, s) = runs
    assert np.array_equal(f, f_ref)
    for k in ("A", "B", "A_RTT", "SI"):
        assert np.array_equal(s[k], s_ref[k]), k
    scale = max(np.abs(s_ref["B"]).max(), 1e-30)
    if name != "none":
        # sums of the box's momentum (about 0.05 a node) in 48-bit pairs
        bar = 1e-12 * scale + 2.0 ** -46 * 0.05 * m.size
        assert np.abs(s["DRTT"] - s_ref["DRTT"]).max() <= bar


def test_a_pass_reports_an_unstable_node(gb):
    # the state blows up within a few steps; the pass's levels raise the flag
    lat = gb.Lattice(np.zeros((64, 256), np.uint8), 0.5000001, 0.45, storage="f16dev")
    lat.set_populations(inputs.random_populations(256, 64, seed=5, lo=0.0, hi=0.6))
    with pytest.raises(gb.LbmError) as e:
        lat.step(1201)
    assert e.value.code == 4
    lat.close()

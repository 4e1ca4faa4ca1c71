"""16-bit storage runs one collision, whatever the extents of the domain."""
import numpy as np
import pytest

from paper_1610_01388_gb300 import lbm
from paper_1610_01388_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, NY = 128, 64


def _tiled(lat, copies, model, storage, layout, newton):
    """A periodic box of `copies` equal tiles along y, cells and populations."""
    rng = np.random.default_rng(4)
    mask = np.tile((rng.random((NY, NX)) < 0.15).astype(np.uint8), (copies, 1))[None]
    s = lbm.Solver(lat, mask, model=model, storage=storage, layout=layout, mu_p=0.08, sigma_y=2e-5,
                   m=1e6, g=(2e-5, -1e-5, 0.0), newton_iters=newton)
    _, w = lbm.lbm_lattice_info(lat)
    f = W.random_populations(w, NY * NX, amplitude=0.01, seed=6).reshape((len(w), 1, NY, NX))
    s.set_populations(np.tile(f, (1, 1, copies, 1)))
    return s


@pytest.mark.parametrize("layout", ["dense", "compact"])
@pytest.mark.parametrize("storage", ["F16", "BF16"])
@pytest.mark.parametrize("model,newton", [("IR", 0), ("PR", 0), ("PR", 2)])
@pytest.mark.parametrize("lat", ["D2Q9", "D3Q15", "D3Q19", "D3Q27"])
def test_a_cell_steps_alike_in_boxes_of_any_extent(lat, model, newton, storage, layout):
    """The first tile of a box of two or four has the cell indices, hence the
    rounding draws, of the tile alone, and the same neighbours: one step leaves
    the same bits in it."""
    one = _tiled(lat, 1, model, storage, layout, newton)
    one.step(1)
    want = one.get_populations()
    for copies in (2, 4):
        s = _tiled(lat, copies, model, storage, layout, newton)
        s.step(1)
        np.testing.assert_array_equal(s.get_populations()[:, :, :NY], want)
        if model == "PR":
            np.testing.assert_array_equal(np.reshape(s.get_tau(), (1, -1, NX))[:, :NY],
                                          np.reshape(one.get_tau(), (1, NY, NX)))
        s.close()
    one.close()


@pytest.mark.parametrize("storage", ["F16", "BF16"])
@pytest.mark.parametrize("model", ["IR", "PR"])
@pytest.mark.parametrize("lat", ["D2Q9", "D3Q15", "D3Q19", "D3Q27"])
def test_a_batch_steps_a_wide_domain_as_a_solver_does(lat, model, storage):
    rng = np.random.default_rng(1)
    mask = (rng.random((1, 130, 131)) < 0.15).astype(np.uint8)
    kw = dict(model=model, storage=storage, mu_p=0.08, sigma_y=2e-5, m=1e6, g=(2e-5, -1e-5, 0.0))
    _, w = lbm.lbm_lattice_info(lat)
    f = W.random_populations(w, mask.size, amplitude=0.01, seed=2).reshape((len(w),) + mask.shape)
    s = lbm.Solver(lat, mask, check_every=100, **kw)
    b = lbm.Batch(1 << 30, check_every=100)
    d = b.add(lat, mask, **kw)
    s.set_populations(f)
    lbm.lbm_set_populations(b.solver(d), f)
    s.step(5)
    b.step(5)
    np.testing.assert_array_equal(lbm.lbm_get_populations(b.solver(d)), s.get_populations())
    s.close()
    b.close()

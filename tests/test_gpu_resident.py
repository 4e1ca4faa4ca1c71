"""Runs of plain steps kept in shared memory (small dense domains) leave the
bits that separate steps leave, and stay near the FP64 oracle."""
import numpy as np
import pytest

from paper_1610_01388_gb300 import lbm
from paper_1610_01388_gb300 import workloads as W
from _pairs import make_pair, rel_l2_u

pytestmark = pytest.mark.gpu

# one warp; a ragged last warp; one full block; several blocks with a ragged
# last one; the largest that fits and the first that does not
SHAPES_2D = [(1, 4, 7), (1, 13, 11), (1, 64, 8), (1, 66, 128), (1, 80, 128), (1, 81, 128)]
SHAPES_3D = [(3, 4, 5), (8, 8, 8), (1, 64, 64), (16, 16, 32), (17, 16, 32)]


def _state(lat, shape, model, storage, **kw):
    rng = np.random.default_rng(5)
    mask = (rng.random(shape) < 0.15).astype(np.uint8)
    s = lbm.Solver(lat, mask, model=model, storage=storage, mu_p=0.08, sigma_y=1e-5, m=1e5,
                   g=(2e-5, -1e-5, 0.0), **kw)
    _, w = lbm.lbm_lattice_info(lat)
    f = W.random_populations(w, mask.size, amplitude=0.01, seed=3)
    s.set_populations(f.reshape((len(w),) + mask.shape))
    return s


def _same(a, b, model):
    fa, fb = a.get_populations(), b.get_populations()
    np.testing.assert_array_equal(fa, fb)
    if model == "PR":
        np.testing.assert_array_equal(a.get_tau(), b.get_tau())


@pytest.mark.parametrize("storage", ["F64", "F32", "F16", "BF16"])
@pytest.mark.parametrize("model", ["IR", "PR"])
@pytest.mark.parametrize("lat,shape", [("D2Q9", s) for s in SHAPES_2D]
                         + [(lat, s) for lat in ("D3Q15", "D3Q19", "D3Q27") for s in SHAPES_3D])
def test_run_equals_single_steps(lat, shape, model, storage):
    a, b = (_state(lat, shape, model, storage) for _ in range(2))
    for n in (4, 5, 23, 64):                  # even and odd runs, one after another
        a.step(n)
        for _ in range(n):
            b.step(1)
        _same(a, b, model)
    a.close()
    b.close()


@pytest.mark.parametrize("kw", [dict(check_every=10), dict(newton_iters=3),
                                dict(flags=lbm.LBM_FLAG_BURNETT_X), dict(flags=lbm.LBM_FLAG_Z_GHOSTS)])
def test_run_with_options_equals_single_steps(kw):
    a, b = (_state("D3Q19", (6, 9, 10), "PR", "F32", **kw) for _ in range(2))
    a.step(37)
    for _ in range(37):
        b.step(1)
    _same(a, b, "PR")
    if "check_every" in kw:
        assert a.residual() == b.residual()
    a.close()
    b.close()


def test_long_run_crosses_launches_and_follows_the_oracle():
    s, o = make_pair("D2Q9", W.channel_mask(4, 32), model="PR", storage="F64", sigma_y=1e-5, m=1e4,
                     g=(1e-5, 0, 0))
    s.step(5000)
    o.step(5000)
    assert s.steps_done == 5000
    assert rel_l2_u(s, o) < 1e-10
    s.close()


def test_table_entry_keeps_its_launch_shape():
    _, _, cls = lbm.lbm_tuning_get_shape("D2Q9", "IR", "F32", 256)
    try:
        a = _state("D2Q9", (1, 32, 8), "IR", "F32")
        a.step(40)
        lbm.lbm_tuning_set("D2Q9", "IR", "F32", cls, 128)
        b = _state("D2Q9", (1, 32, 8), "IR", "F32")
        b.step(40)
        _same(a, b, "IR")
    finally:
        lbm.lbm_tuning_clear()


@pytest.mark.parametrize("model", ["IR", "PR"])
@pytest.mark.parametrize("lat,shape", [("D2Q9", (1, 13, 11)), ("D2Q9", (1, 33, 31)), ("D2Q9", (1, 79, 80)),
                                       ("D3Q15", (5, 6, 7)), ("D3Q15", (20, 21, 19)),
                                       ("D3Q19", (5, 6, 7)), ("D3Q19", (15, 16, 17)),
                                       ("D3Q27", (5, 6, 7)), ("D3Q27", (15, 16, 17))])
@pytest.mark.parametrize("flags", [0, lbm.LBM_FLAG_BURNETT_X, lbm.LBM_FLAG_Z_GHOSTS])
def test_divided_fp64_steps_equal_undivided_ones(lat, shape, model, flags):
    """Small FP64 domains divide a cell's work over warps; a table entry keeps
    the undivided kernel.  Same expressions, same bits."""
    if flags == lbm.LBM_FLAG_Z_GHOSTS and lat == "D2Q9":
        pytest.skip("ghost planes need a 3D lattice")
    _, _, cls = lbm.lbm_tuning_get_shape(lat, model, "F64", int(np.prod(shape)))
    try:
        a = _state(lat, shape, model, "F64", flags=flags)
        a.step(3)                         # single steps
        a.step(21)                        # a run
        lbm.lbm_tuning_set(lat, model, "F64", cls, 128)
        b = _state(lat, shape, model, "F64", flags=flags)
        b.step(24)
        _same(a, b, model)
    finally:
        lbm.lbm_tuning_clear()

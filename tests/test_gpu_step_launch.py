"""How plain steps are launched does not change what they compute: a run of
steps queued at once (overlapped launches, graphs) leaves the same bits as the
same steps taken one at a time with a wait after each."""
import numpy as np
import pytest

from paper_1610_01388_gb300 import lbm
from paper_1610_01388_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    # lattice, model, storage, layout, mask: one block, a ragged last warp, one
    # wave, many waves
    ("D2Q9", "IR", "F64", "dense", lambda: W.channel_mask(4, 64)),
    ("D2Q9", "PR", "F16", "dense", lambda: W.channel_mask(33, 19)),
    ("D3Q15", "PR", "F32", "dense", lambda: W.porous_mask((37, 29, 23), 0.7, 3, 5, seed=4)[0]),
    ("D3Q19", "IR", "F16", "compact", lambda: W.porous_mask(40, 0.7, 3, 5, seed=4)[0]),
    ("D3Q19", "PR", "F32", "compact", lambda: W.porous_mask(40, 0.7, 3, 5, seed=4)[0]),
    ("D3Q27", "PR", "BF16", "dense", lambda: W.duct_mask(130, 65, 64)),
    ("D3Q27", "IR", "F32", "dense", lambda: W.duct_mask(130, 65, 64)),
]


def _solver(lat, mask, model, storage, layout, check_every):
    s = lbm.Solver(lat, mask, model=model, storage=storage, layout=layout, mu_p=0.08, sigma_y=1e-5,
                   m=1e5, g=(2e-5, 0.0, 0.0), check_every=check_every)
    _, w = lbm.lbm_lattice_info(lat)
    f = W.random_populations(w, mask.size, amplitude=0.01, seed=3)
    s.set_populations(f.reshape((len(w),) + mask.shape))
    return s


@pytest.mark.parametrize("check_every", [0, 37])
@pytest.mark.parametrize("lat,model,storage,layout,make", CASES)
def test_queued_steps_equal_waited_steps(lat, model, storage, layout, make, check_every):
    mask = make()
    a = _solver(lat, mask, model, storage, layout, check_every)
    b = _solver(lat, mask, model, storage, layout, check_every)
    a.step(150)
    for _ in range(150):
        b.step(1)
        b.sync()
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    if model == "PR":
        np.testing.assert_array_equal(a.get_tau(), b.get_tau())
    if check_every:
        assert a.residual() == b.residual()
    a.close()
    b.close()


@pytest.mark.parametrize("check_every", [0, 7])
@pytest.mark.parametrize("lat,model,storage,shape", [
    # steps that fill more than half the GPU and less than all of it, in both
    # layouts, and the sizes around: overlapped, plain, overlapped launches
    ("D3Q15", "PR", "F32", (40, 40, 40)), ("D3Q15", "PR", "F32", (48, 48, 48)),
    ("D3Q15", "PR", "F32", (64, 64, 64)), ("D3Q27", "IR", "F16", (48, 48, 48)),
    ("D3Q27", "IR", "F16", (64, 64, 64)), ("D2Q9", "IR", "F32", (1, 400, 512)),
    ("D3Q19", "PR", "F64", (20, 33, 33))])
@pytest.mark.parametrize("layout", ["dense", "compact"])
def test_overlapped_and_plain_launches_leave_the_same_bits(lat, model, storage, shape, layout, check_every):
    rng = np.random.default_rng(6)
    mask = (rng.random(shape) < 0.2).astype(np.uint8)
    a, b = (_solver(lat, mask, model, storage, layout, check_every) for _ in range(2))
    a.step(40)
    for _ in range(40):
        b.step(1)
        b.sync()
    np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    if check_every:
        assert a.residual() == b.residual()
    a.close()
    b.close()

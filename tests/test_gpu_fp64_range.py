"""FP64 steps over the whole range of their arithmetic: the reciprocals and roots
of the FP64 collision have no shorter range than a division and a square root."""
import numpy as np
import pytest

from paper_1610_01388_gb300 import lbm
from paper_1610_01388_gb300 import workloads as W
from _pairs import gpu_to_oracle, make_pair, set_both

pytestmark = pytest.mark.gpu

SHAPES = {"D2Q9": (1, 6, 11), "D3Q15": (5, 6, 7), "D3Q19": (5, 6, 7), "D3Q27": (5, 6, 7)}


@pytest.mark.parametrize("steps", [[1] * 12, [12]])     # single steps; a run
@pytest.mark.parametrize("lat", sorted(SHAPES))
def test_newtonian_creep_is_linear_in_its_force(lat, steps):
    """Without a yield stress a creeping flow is proportional to its force: one
    2^382 times weaker, whose squared stress lies near 2^-964, has velocities
    2^382 times smaller.  Only a stress whose square underflows (below 2^-537,
    2^-55 of the force) counts as none: 12 steps of at most 27 such terms."""
    mask = np.zeros(SHAPES[lat], np.uint8)
    mask[:, 0] = 1
    u = []
    for e in (100, 482):
        s = lbm.Solver(lat, mask, model="IR", storage="F64", mu_p=0.1, sigma_y=0.0,
                       g=(2.0 ** -e, 0.0, 0.0))
        for n in steps:
            s.step(n)
        u.append(s.fields()[1][0] * 2.0 ** e)
        s.close()
    assert u[0].max() > 1.0
    np.testing.assert_allclose(*u, rtol=0, atol=12 * 27 * 2.0 ** -55)


@pytest.mark.parametrize("m,sigma_y,magic", [(1e300, 1e-6, 0.25), (1e300, 1e6, 0.25), (5e307, 1.0, 0.25),
                                             (1e4, 1e-5, 1e300), (1e20, 1.0, 1e300)])
@pytest.mark.parametrize("lat", sorted(SHAPES))
def test_extreme_relaxation_times(lat, m, sigma_y, magic):
    """An extreme regularisation makes tau 3e294, 3e306 or 1.5e308 (its reciprocal
    is subnormal): the even rate vanishes, the odd one does not, and 1 / rho is
    unharmed.  An extreme magic number does it to the odd rate.  The FP64 oracle
    within rounding."""
    mask = np.zeros(SHAPES[lat], np.uint8)
    mask[:, 0] = 1
    s, o = make_pair(lat, mask, model="PR", storage="F64", sigma_y=sigma_y, m=m, magic=magic,
                     g=(1e-5, 0, 0))
    _, w = lbm.lbm_lattice_info(lat)
    f = W.random_populations(w, mask.size, amplitude=0.01, seed=3)
    set_both(lat, s, o, gpu_to_oracle(lat, f.reshape((len(w),) + mask.shape)))
    s.step(3)
    o.step(3)
    fluid = mask.reshape(-1) == 0
    got = gpu_to_oracle(lat, s.get_populations())[:, fluid]
    want = o.f[:, fluid]
    assert np.all(np.isfinite(want))
    # three collisions of O(100) operations on numbers below 1/2
    np.testing.assert_allclose(got, want, rtol=0, atol=3 * 100 * 2.0 ** -54)
    s.close()

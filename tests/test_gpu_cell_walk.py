"""The sweeps of a case without a list: each lane puts its hits aside and
evaluates them when its places run out.  The number of places follows the
block size, so the bits may not depend on it; against the list the sums differ
by their order only (1e-12 of the field's maximum in FP64, 1e-4 in FP32 after
two advection steps)."""
import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")


def fields(case, dim, precision, **kw):
    h = S.case_from_spec(case, precision=precision, **kw)
    S.step(h, 2)
    out = [S.read_fields(h, f, dim) for f in (S.FIELD_POS, S.FIELD_VEL, S.FIELD_GRADC, S.FIELD_ACC_VISC)]
    S.destroy(h)
    return out


# neighbours per particle: fewer than the 20 places of the narrowest sweep,
# about the 56 of the widest, and several times as many (18 candidates a cell
# to 110, so a cell is read in 2 to 7 steps)
@pytest.mark.parametrize("dim,h_factor", [(2, 1.3), (2, 2.2), (2, 5.0), (3, 1.0), (3, 1.3), (3, 2.4)])
@pytest.mark.parametrize("precision", [32, 64])
def test_the_bits_do_not_follow_the_places(dim, h_factor, precision):
    case = sphcases.small_droplet(dim, 26 if dim == 2 else 12, seed=4, jitter=0.1, vel_amp=0.02)
    case.h_factor = h_factor
    a = fields(case, dim, precision, nbr_mode=S.NBR_CELLS, block=32)
    for block in (160, 256):
        for x, y in zip(a, fields(case, dim, precision, nbr_mode=S.NBR_CELLS, block=block)):
            assert np.array_equal(x, y)
    for x, y in zip(a, fields(case, dim, precision, max_neighbors=1000)):
        assert np.abs(x - y).max() <= (1e-12 if precision == 64 else 1e-4) * np.abs(y).max()

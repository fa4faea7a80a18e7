"""FP64 engines take smaller blocks than asked for until every SM has eight:
below that size all blocks asked for are the same launch.  These cases are large
enough, at 8 lanes per particle, to run in the blocks they ask for, and none
changes a bit, with the pair geometry stored or not."""
import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")
FIELDS = (S.FIELD_POS, S.FIELD_VEL, S.FIELD_RHO, S.FIELD_GRADC, S.FIELD_ACC_VISC)


def fields(case, block, keep, **kw):
    h = S.case_from_spec(case, precision=64, block=block, lanes=8, **kw)
    S.set_pair_geometry(h, keep)
    S.step(h, 1)
    out = [S.read_fields(h, f, case.dim) for f in FIELDS]
    S.destroy(h)
    return out


@pytest.mark.parametrize("dim,n_side", [(2, 204), (3, 35)])
@pytest.mark.parametrize("nbr_mode", [S.NBR_LIST, S.NBR_CELLS])
def test_the_bits_do_not_follow_the_block(dim, n_side, nbr_mode):
    case = sphcases.small_droplet(dim, n_side, seed=4, jitter=0.1, vel_amp=0.02)
    assert case.n_fluid * 8 >= S.device_info()["sm_count"] * 8 * 256
    want = fields(case, 32, True, nbr_mode=nbr_mode)
    for block, keep in ((64, True), (96, False), (160, True), (256, True), (256, False)):
        for x, y in zip(fields(case, block, keep, nbr_mode=nbr_mode), want):
            assert np.array_equal(x, y)

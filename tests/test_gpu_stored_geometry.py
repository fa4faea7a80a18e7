"""FP64 list cases read the pair geometry of their lists from memory and run
in blocks made smaller for small cases; the cell walk computes the same
geometry for every pair.  The two differ by the order of the sums: 1e-12 of
each field's maximum after two advection steps (the bar of the list against
the walk), at 1 to 8 lanes (odd list parts per lane), a list that crosses 32
slots by one, walls, and a periodic axis."""
import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")


def cases():
    return {"walls_2d": sphcases.small_droplet(2, 21, seed=4, jitter=0.1, vel_amp=0.05),
            "walls_3d": sphcases.small_droplet(3, 11, seed=5, jitter=0.1, vel_amp=0.05),
            "periodic_3d": sphcases.periodic_blob(3, 14, seed=6),
            "few_2d": sphcases.free_blob(2, 7, seed=8, rho_ratio=10.0)}


@pytest.mark.parametrize("lanes,block", [(1, 256), (2, 96), (4, 64), (8, 32)])
@pytest.mark.parametrize("name", sorted(cases()))
def test_stored_geometry_agrees_with_the_walk(name, lanes, block):
    case = cases()[name]
    out = []
    for kw in (dict(nbr_mode=S.NBR_CELLS), dict(lanes=lanes, block=block)):
        h = S.case_from_spec(case, precision=64, **kw)
        info = S.step(h, 2)
        out.append([S.read_fields(h, f, case.dim) for f in (S.FIELD_VEL, S.FIELD_GRADC, S.FIELD_ACC_VISC, S.FIELD_PRESSURE)]
                   + [info["n_sub"]])
        S.destroy(h)
    assert out[0][-1] == out[1][-1]
    for a, b in zip(out[0][:-1], out[1][:-1]):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()

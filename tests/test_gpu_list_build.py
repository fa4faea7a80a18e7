"""The neighbour-list build at its edges: cells whose surroundings hold more
candidates than the build stages at a time, cells with more slots than one
group of shared lists, odd capacities, and capacities that just fit.  The
list and the cell walk hold the same neighbours and differ by the order of
the sums only, so the bars are those of the list against the walk: 1e-12 of
the field's maximum in FP64, 1e-4 in FP32 after two advection steps."""
import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")


def fields(case, dim, precision, **kw):
    h = S.case_from_spec(case, precision=precision, **kw)
    info = S.step(h, 2)
    out = [S.read_fields(h, f, dim) for f in (S.FIELD_VEL, S.FIELD_GRADC, S.FIELD_ACC_VISC)]
    counts = S.debug_neighbor_counts(h)
    S.destroy(h)
    return out, info["n_sub"], counts


@pytest.mark.parametrize("dim,h_factor,cap", [(2, 1.3, 33), (2, 2.2, 97), (2, 5.0, 400), (3, 1.3, 127), (3, 1.9, 400),
                                              (3, 2.4, 1000)])
@pytest.mark.parametrize("precision", [32, 64])
def test_crowded_cells_agree_with_the_walk(dim, h_factor, cap, precision):
    # h_factor raises the particles per cell: 2D 7 to 100, 3D 18 to 110
    # (27 x 110 candidates, 5 stages), list capacities odd and even
    case = sphcases.small_droplet(dim, 26 if dim == 2 else 12, seed=3, jitter=0.1, vel_amp=0.02)
    case.h_factor = h_factor
    a, na, counts = fields(case, dim, precision, max_neighbors=cap)
    b, nb, _ = fields(case, dim, precision, nbr_mode=S.NBR_CELLS)
    assert counts.max() <= cap and na == nb
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= (1e-12 if precision == 64 else 1e-4) * np.abs(y).max()


@pytest.mark.parametrize("precision", [32, 64])
def test_a_capacity_that_just_fits_is_accepted(precision):
    # on the lattice 2h = 3 dx, so a whole shell of particles lies at 2h to
    # rounding; the largest neighbour count is enough capacity, one less is not
    case = sphcases.small_droplet(3, 10)
    case.h_factor = 1.5
    h = S.case_from_spec(case, precision=precision, nbr_mode=S.NBR_CELLS, max_substeps=1)
    S.step(h, 1, check=False)
    kind = case.flat()[3]
    most = int(S.debug_neighbor_counts(h)[kind < 2].max())
    S.destroy(h)
    for cap, ok in ((most, True), (most - 1, False)):
        h = S.case_from_spec(case, precision=precision, max_neighbors=cap, max_substeps=1)
        rc = S.step(h, 1, check=False)["rc"]
        S.destroy(h)
        assert (rc != S.ERR_NEIGHBORS) == ok

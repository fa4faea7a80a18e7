"""In the cell walk two lanes share a particle, or one thread takes it where the
engine's particles fill the GPU; the two sum in the same order.  So a small
case has the same bits alone (two lanes) and in a batch that a large case
fills, and the large case the same as walked by its list's neighbours to the
rounding of a reordered sum (1e-4 in FP32, 1e-12 in FP64, of each field's
maximum)."""
import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")
FIELDS = (S.FIELD_POS, S.FIELD_VEL, S.FIELD_RHO, S.FIELD_GRADC, S.FIELD_ACC_VISC)


def read(h, dim):
    return [S.read_fields(h, f, dim) for f in FIELDS]


# particles per SM from which each sweep takes one thread: 1024 (A) and 2048
# in FP32, 512 (A in 3D) in FP64; the sizes lie on either side on 152 SMs
@pytest.mark.parametrize("dim,precision,n_side", [(2, 32, 420), (2, 32, 570), (3, 32, 56), (3, 32, 69), (3, 64, 44)])
def test_the_bits_do_not_follow_the_population(dim, precision, n_side):
    small = {"walls": sphcases.small_droplet(dim, 21 if dim == 2 else 11, seed=4, jitter=0.1, vel_amp=0.02),
             "periodic": sphcases.periodic_blob(dim, 17 if dim == 2 else 13, seed=6)}
    alone = {}
    for name, case in small.items():
        h = S.case_from_spec(case, precision=precision, nbr_mode=S.NBR_CELLS)
        S.step(h, 1)
        alone[name] = read(h, dim)
        S.destroy(h)
    large = sphcases.small_droplet(dim, n_side, seed=7, jitter=0.1, vel_amp=0.02)
    hs = {"large": S.case_from_spec(large, precision=precision, nbr_mode=S.NBR_CELLS)}
    for name, case in small.items():
        hs[name] = S.case_from_spec(case, precision=precision, nbr_mode=S.NBR_CELLS)
    batch = S.batch_create(precision)
    for h in hs.values():
        S.batch_add(batch, h)
    S.batch_step(batch, 1)
    got = {name: read(h, dim) for name, h in hs.items()}
    for h in hs.values():
        S.batch_remove(batch, h)
        S.destroy(h)
    S.batch_destroy(batch)
    for name in small:
        for x, y in zip(got[name], alone[name]):
            assert np.array_equal(x, y)
    h = S.case_from_spec(large, precision=precision)
    S.step(h, 1)
    for k, (x, y) in enumerate(zip(got["large"], read(h, dim))):
        if FIELDS[k] == S.FIELD_POS:
            x, y = x - large.flat()[0][:, :dim], y - large.flat()[0][:, :dim]
        if FIELDS[k] == S.FIELD_RHO:
            x, y = x - np.round(x), y - np.round(y)
        assert np.abs(x - y).max() <= (1e-12 if precision == 64 else 1e-4) * np.abs(y).max()
    S.destroy(h)

"""A case does not know its unit of length.  Scaled by a power of two (with
c0, velocities, viscosity and surface tension to match, time unchanged) every
operation scales exactly, so the results are the same bits after scaling back,
as long as nothing leaves the type's range.  The scales below keep h within
the range of the kernel's constants (FP32: -5 alpha_d / h finite in 3D down to
h = 2.8e-10, in 2D down to 2e-13); densities are scaled by the reciprocal, so
that products of two viscosities stay normal numbers too."""
import dataclasses

import numpy as np
import pytest

import sphcases

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2503_16082_gb300")


def scaled(case, s):
    phases = [dataclasses.replace(p, pos=p.pos * s, rho0=p.rho0 / s, eta=p.eta * s, vel=None if p.vel is None else p.vel * s)
              for p in case.phases]
    return dataclasses.replace(case, lo=[x * s for x in case.lo], hi=[x * s for x in case.hi], dx=case.dx * s,
                               c0=case.c0 * s, gamma=case.gamma * s**2, phases=phases)


def fields(case, precision, s, steps=2, **kw):
    h = S.case_from_spec(scaled(case, s), precision=precision, **kw)
    info = S.step(h, steps, check=False)
    unit = {S.FIELD_POS: s, S.FIELD_VEL: s, S.FIELD_RHO: 1.0 / s, S.FIELD_GRADC: 1.0 / s, S.FIELD_ACC_VISC: s}
    out = [S.read_fields(h, f, case.dim) / u for f, u in unit.items()]
    q = S.diagnose(h, center=[0.5 * s] * case.dim)
    out.append(np.array(q["momentum"]) / s**case.dim)
    S.destroy(h)
    return info["rc"], info["n_sub"], out


@pytest.mark.parametrize("dim,precision,exponent", [(3, 32, -28), (2, 32, -36), (3, 32, 20), (3, 64, -50)])
@pytest.mark.parametrize("nbr_mode", [S.NBR_LIST, S.NBR_CELLS])
def test_the_bits_do_not_follow_the_unit_of_length(dim, precision, exponent, nbr_mode):
    case = sphcases.small_droplet(dim, 20 if dim == 2 else 12, seed=2, jitter=0.1, vel_amp=0.02)
    rc0, n0, a = fields(case, precision, 1.0, nbr_mode=nbr_mode)
    rc1, n1, b = fields(case, precision, 2.0**exponent, nbr_mode=nbr_mode)
    assert (rc0, rc1) == (S.OK, S.OK) and n0 == n1
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("exponent", [-100, 62, 100])
def test_fp64_lists_hold_beyond_the_range_of_fp32(dim, exponent):
    # the list build tests candidates in FP32 first: lengths whose squares
    # FP32 cannot hold, and lengths around 1e18
    case = sphcases.small_droplet(dim, 20 if dim == 2 else 12, seed=2, jitter=0.1, vel_amp=0.02)
    rc0, n0, a = fields(case, 64, 1.0)
    rc1, n1, b = fields(case, 64, 2.0**exponent)
    assert (rc0, rc1) == (S.OK, S.OK) and n0 == n1
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("nbr_mode", [S.NBR_LIST, S.NBR_CELLS])
@pytest.mark.parametrize("second", [0, 1])
def test_fp32_pair_whose_squared_distance_is_denormal(nbr_mode, second):
    # two fluid particles 2^-38 apart next to a cell's corner (h = 1/4, so the
    # grid's lines are exact), among their neighbours: scaled by 2^-28 their
    # r^2 = 2^-132 is a denormal.  Finite, and the same results: the pair's e_ij
    # is weighed by W' or r everywhere but in the penalty, where 1/r is taken in
    # full, so its error stays below the rounding of a sum (2^-24 of its terms);
    # the bar is 16 of these after one step, of each field's maximum (in a second
    # one the offsets, no longer next to the corner, would round together)
    cs = 0.5 * (1 + 2.0**-16)
    corner = 4 * cs
    rng = np.random.default_rng(3)
    p = sphcases.lattice([0.0, 0.0], [4.0, 4.0], 0.25) + rng.uniform(-0.02, 0.02, (256, 2))
    p = p[np.abs(p - corner).max(axis=1) > 0.2]
    p = np.concatenate([[[0.0, 0.0]], p[(p > 0.05).any(axis=1)], [[corner, corner], [corner + 2.0**-38, corner]]])
    kind = np.hypot(*(p - corner).T) < 0.8
    kind[-1] = not second
    phases = [sphcases.Phase("fluid", p[k], rho0=r, eta=0.1, vel=np.full((k.sum(), 2), 0.01)) for k, r in ((kind, 2.0), (~kind, 1.0))]
    case = sphcases.Case(name="close", dim=2, lo=[0.0, 0.0], hi=[4.0, 4.0], dx=0.25, gamma=1.0, c0=10.0, h_factor=1.0, phases=phases)
    rc0, n0, a = fields(case, 32, 1.0, steps=1, nbr_mode=nbr_mode)
    rc1, n1, b = fields(case, 32, 2.0**-28, steps=1, nbr_mode=nbr_mode)
    assert (rc0, rc1) == (S.OK, S.OK) and n0 == n1
    for x, y in zip(a[:5], b[:5]):
        assert np.isfinite(x).all() and np.abs(x - y).max() <= 2.0**-20 * np.abs(x).max()

"""The stored pair geometry of FP64 lists: counted in the footprint, and worth
no bit of any result."""
import numpy as np
import pytest

import sphcases

S = pytest.importorskip("paper_2503_16082_gb300")
from paper_2503_16082_gb300 import serve


def params(precision=64, **kw):
    return S.default_params(dim=3, precision=precision, dx=0.01, **kw)


def test_the_footprint_counts_the_geometry():
    n, k = 100_000, 128
    listed = S.footprint_bytes(params(), n) - S.footprint_bytes(params(nbr_mode=S.NBR_CELLS), n)
    assert listed >= n * k * (4 + 48)
    assert S.pair_geometry_bytes(params(), n) == n * k * 48
    assert S.pair_geometry_bytes(params(), 33) == 64 * k * 48                  # rows of 32 slots
    assert S.pair_geometry_bytes(params(max_neighbors=100), 32) == 32 * 100 * 48
    assert S.pair_geometry_bytes(params(32), n) == 0
    assert S.pair_geometry_bytes(params(nbr_mode=S.NBR_CELLS), n) == 0
    # a case whose geometry is more than an engine keeps goes without
    most = (16 << 30) // (48 * k) // 32 * 32
    assert 0 < S.pair_geometry_bytes(params(), most) <= 16 << 30
    assert S.pair_geometry_bytes(params(), most + 1) == 0
    assert S.footprint_bytes(params(), most + 1) < S.footprint_bytes(params(), most)


def test_a_request_too_large_with_its_geometry_goes_without():
    srv = serve.Server(precision=64)
    spec = sphcases.small_droplet(3, 10)
    full = srv.footprint(spec)
    least = full - S.pair_geometry_bytes(srv._params(spec), spec.n)
    for budget, refused, keep in ((full, False, True), (full - 1, False, False), (least, False, False), (least - 1, True, None)):
        srv.budget = budget
        f = srv.submit(spec, n_adv=1)
        assert f.done() == refused
        if not refused:
            r = srv.queue.pop()
            assert r.keep_geometry == keep and r.footprint == (full if keep else least) <= budget


@pytest.mark.gpu
@pytest.mark.parametrize("keep", [True, False])
def test_an_engine_takes_no_more_than_its_footprint(keep):
    import torch

    case = sphcases.small_droplet(3, 34, seed=3, jitter=0.1)
    warm = S.case_from_spec(sphcases.small_droplet(2, 12), precision=64)
    S.step(warm, 1)
    p = S.params_from_spec(case, 64)
    bound = S.footprint_bytes(p, case.n) - (0 if keep else S.pair_geometry_bytes(p, case.n))
    h = S.case_from_spec(case, precision=64)
    S.set_pair_geometry(h, keep)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    S.step(h, 0)
    torch.cuda.synchronize()
    # 32 MB for the captured graph and the allocation granularity; the geometry is 240 MB
    assert before - torch.cuda.mem_get_info()[0] <= bound + (32 << 20)
    with pytest.raises(S.SphstError):
        S.set_pair_geometry(h, True)
    S.destroy(h)
    S.destroy(warm)


def cases():
    return {"walls_2d": sphcases.small_droplet(2, 21, seed=4, jitter=0.1, vel_amp=0.05),
            "walls_3d": sphcases.small_droplet(3, 11, seed=5, jitter=0.1, vel_amp=0.05),
            "periodic_3d": sphcases.periodic_blob(3, 14, seed=6),
            "few_2d": sphcases.free_blob(2, 7, seed=8, rho_ratio=10.0)}


FIELDS = (S.FIELD_POS, S.FIELD_VEL, S.FIELD_RHO, S.FIELD_GRADC, S.FIELD_ACC_VISC)


@pytest.mark.gpu
@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("name", sorted(cases()))
@pytest.mark.parametrize("corr", [0, 1])
def test_the_bits_do_not_follow_the_geometry(lanes, name, corr):
    case = cases()[name]
    out = []
    for keep in (True, False):
        h = S.case_from_spec(case, precision=64, lanes=lanes, surface_corr=corr)
        S.set_pair_geometry(h, keep)
        S.step(h, 2)
        out.append([S.read_fields(h, f, case.dim) for f in FIELDS])
        S.destroy(h)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("work_lists", [0, 1])
def test_a_batch_holds_members_with_and_without(work_lists):
    alone, batch, hs = [], S.batch_create(64), []
    for k, name in enumerate(sorted(cases())):
        case = cases()[name]
        h = S.case_from_spec(case, precision=64)
        S.step(h, 2)
        alone.append([S.read_fields(h, f, case.dim) for f in FIELDS])
        S.destroy(h)
        hs.append(S.case_from_spec(case, precision=64, work_lists=work_lists))
        S.set_pair_geometry(hs[-1], k % 2 == 1)
        S.batch_add(batch, hs[-1])
    S.batch_step(batch, 2)
    for h, name, want in zip(hs, sorted(cases()), alone):
        for f, x in zip(FIELDS, want):
            assert np.array_equal(S.read_fields(h, f, cases()[name].dim), x)
        S.batch_remove(batch, h)
        S.destroy(h)
    S.batch_destroy(batch)


@pytest.mark.gpu
@pytest.mark.parametrize("partner", ["wall", "fluid"])
def test_pairs_at_the_cutoff_keep_their_kind(partner):
    # isolated pairs at 2h less a few units in the last place: 1 - q/2 rounds
    # to 0 or to either side of it, so W' is 0 or about 1e-48 and of either sign
    # by the formula.  The pair's sums are that one term, which tells a wall
    # partner (viscosity eta_i, volume dp^2) from a fluid one
    dx = 0.139                          # 0.5 / h rounds up, so one pair in six is past 2h by 1 - q/2
    h = 1.3 * dx
    n = 400
    a = np.stack(np.meshgrid(np.arange(20.0), np.arange(20.0), indexing="ij"), axis=-1).reshape(-1, 2) * (8 * h)
    ang = np.linspace(0.05, 3.0, n)
    b = a + 2 * h * (1 - np.arange(n)[:, None] % 8 * 2.0**-53) * np.stack([np.cos(ang), np.sin(ang)], axis=1)
    phases = [sphcases.Phase("fluid", a, rho0=1.0, eta=0.1, vel=np.full((n, 2), 0.01)),
              sphcases.Phase("fluid", np.array([[-8 * h, -8 * h]]), rho0=3.0, eta=0.01),
              sphcases.Phase("wall", b) if partner == "wall" else sphcases.Phase("wall", np.array([[-8 * h, 0.0]]))]
    if partner == "fluid":
        phases[1].pos = np.concatenate([phases[1].pos, b])
    case = sphcases.Case(name="cutoff", dim=2, lo=[-8 * h] * 2, hi=[160 * h] * 2, dx=dx, gamma=0.0, c0=10.0, phases=phases)
    out, held = [], []
    for keep in (True, False):
        c = S.case_from_spec(case, precision=64)
        S.set_pair_geometry(c, keep)
        S.step(c, 1)
        held.append(S.debug_neighbors(c)[0].sum())
        out.append([S.read_fields(c, f, 2) for f in FIELDS])
        S.destroy(c)
    assert held[0] == held[1] > 50
    assert (np.abs(out[0][4][:n]) > 0).any() and np.abs(out[0][4][:n]).max() < 1e-30
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.gpu
def test_a_profiled_step_counts_its_launches():
    # rebuild: 8 of the cell order, 5 of the slots, then per list class the
    # lists, the stored geometry (FP64) and the band
    case = sphcases.small_droplet(2, 16, seed=3, jitter=0.1)
    want = {(32, S.NBR_LIST, True): 15, (64, S.NBR_LIST, True): 16, (64, S.NBR_LIST, False): 15, (64, S.NBR_CELLS, True): 13}
    for (precision, mode, keep), n in want.items():
        h = S.case_from_spec(case, precision=precision, nbr_mode=mode)
        S.set_pair_geometry(h, keep)
        assert S.profile_step(h)["rebuild"][1] == n
        S.destroy(h)

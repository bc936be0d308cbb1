"""The batch's packed sweeps over operator tables: more than eight members in one group of tables, so that those with
few work items share a launch a sweep.  Every member must match its standalone run bit for bit."""
import numpy as np
import pytest

import paper_2302_12519_gb300 as ep
import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = (ep.EP_V, ep.EP_W, ep.EP_VE, ep.EP_TACT)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2302_12519_gb300 import build
    build.build()
    ep.load()


def _case(seed, nx, ny, nz, kind):
    rng = np.random.default_rng(seed)
    mask = np.ones((nz, ny, nx), np.uint8) if kind == "full" else (rng.random((nz, ny, nx)) > 0.03).astype(np.uint8)
    if kind == "layers":
        z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
        mask = ((x + 0.7 * y + 0.4 * z) / 6.0 % 1.0 < 0.57).astype(np.uint8)
    return W.random_case(seed, nx, ny, nz, model=W.BI, mask=mask)


def _handles(cases):
    out = []
    for i, c in enumerate(cases):
        s = ep.sim_from_case(c)
        s.set_state(*W.random_state(900 + i, c), 3)
        out.append(s)
    return out


# Ten members over rows (4 096 to 9 216 voxels: a last CTA of every fill), two below the 4 096 voxels from which a handle
# has tables (a box, all of it clear items, and one with holes, without any), and with bricks one of 800 thousand voxels
# in thin layers; with 32 planes a work item it has 210 of them, few enough to be packed.
@pytest.mark.parametrize("capped", [False, True])
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("bricks", [False, True])
def test_packed_members_same_alone_and_in_the_mix(bricks, solver, capped):
    cases = [_case(40, 16, 16, 16, "full"), _case(41, 31, 17, 8, "full"), _case(42, 96, 96, 1, "full")]
    cases += [_case(43 + i, 18 + i, 20 + i, 15 - i % 3, "holes") for i in range(7)]
    cases += [_case(51, 13, 11, 9, "full"), _case(52, 15, 14, 13, "holes")]   # clear items only, none
    if bricks:
        cases.append(_case(53, 90, 98, 160, "layers"))
    for c in cases:
        c.params.solver = solver
        if capped:
            c.params.max_iter, c.params.rel_tol, c.params.check_every = 7, 0.0, 3
        elif bricks:   # the large block would take thousands of sweeps from a random state
            c.params.rel_tol = 1e-2
    steps = 12 if capped else 2
    alone, mixed = _handles(cases), _handles(cases)
    b = ep.Batch(len(cases))
    b.set_schedule(0, 32, 0)
    slots = [b.add(s) for s in mixed]
    for s in alone:
        s.step(steps, allow_noconv=True)
    info = b.info()
    assert info.groups == 1 and info.solo_members == 0
    b.step(1, allow_noconv=True)
    b.step(steps - 1, allow_noconv=True)
    for s_alone, s_mix, slot in zip(alone, mixed, slots):
        st = b.slot_stats(slot)
        assert st.step == 3 + steps and (not capped or st.iters == 7)
        for f in FIELDS:
            np.testing.assert_array_equal(s_mix.read(f), s_alone.read(f))
    b.close()
    for s in alone + mixed:
        s.close()


def test_autotune_with_tables_keeps_the_solve():
    """Trial sweeps over rows and bricks leave the members' state as it was."""
    cases = [_case(60, 17, 16, 16, "full"), _case(61, 90, 98, 160, "layers"), _case(62, 13, 11, 9, "full")]
    for c in cases:
        c.params.max_iter, c.params.rel_tol = 5, 0.0
    hs = _handles(cases)
    before = [[s.read(f) for f in FIELDS] for s in hs]
    b = ep.Batch(3)
    for s in hs:
        b.add(s)
    b.autotune(4)
    for s, want in zip(hs, before):
        for f, x in zip(FIELDS, want):
            np.testing.assert_array_equal(s.read(f), x)
    b.step(2, allow_noconv=True)
    assert all(b.slot_stats(i).iters == 5 and b.slot_stats(i).step == 5 for i in range(3))
    b.close()
    for s in hs:
        s.close()


# Two blocks of 64^3 (29 MB of rows each) share a group of at most 60 MB; so do two members with 57 MB of bricks, which
# count half, and two with 37 MB of rows (up to 75 MB a pair); a third joins none of them
@pytest.mark.parametrize("n,size,kind,groups", [(4, (64, 64, 64), "full", 2), (2, (90, 98, 160), "layers", 1),
                                                (3, (90, 98, 160), "layers", 2), (3, (75, 90, 85), "layers", 2)])
def test_members_that_share_a_group(n, size, kind, groups):
    cases = [_case(80 + i, *size, kind) for i in range(n)]
    for c in cases:
        c.params.solver, c.params.max_iter, c.params.rel_tol, c.params.check_every = 1, 6, 0.0, 4
    alone, mixed = _handles(cases), _handles(cases)
    b = ep.Batch(n)
    for s in mixed:
        b.add(s)
    assert b.info().groups == groups
    b.step(2, allow_noconv=True)
    for a, m in zip(alone, mixed):
        a.step(2, allow_noconv=True)
        for f in FIELDS:
            np.testing.assert_array_equal(m.read(f), a.read(f))
    b.close()
    for s in alone + mixed:
        s.close()


# Members of 32 and 34 sweep CTAs of rows go one, two and three to a CTA of the packed launch; 912 CTAs are resident on
# 152 SMs
@pytest.mark.parametrize("n", [40, 60, 100])
def test_packed_ctas_that_take_several_sweep_ctas(n):
    cases = [_case(100 + i % 7, 32, 8, 16 + i % 2, "full") for i in range(n)]
    for i, c in enumerate(cases):
        c.params.max_iter, c.params.rel_tol, c.params.check_every = 5 + 3 * (i % 3), 0.0, 4
    alone, mixed = _handles(cases), _handles(cases)
    b = ep.Batch(n)
    for s in mixed:
        b.add(s)
    assert b.info().solo_members == 0 and b.info().groups == 1
    b.step(2, allow_noconv=True)
    for a, m in zip(alone, mixed):
        a.step(2, allow_noconv=True)
        for f in FIELDS:
            np.testing.assert_array_equal(m.read(f), a.read(f))
    b.close()
    for s in alone + mixed:
        s.close()

"""Batched monodomain members over operator tables: every member must match its standalone run bit for bit."""
import numpy as np
import pytest

import paper_2302_12519_gb300 as ep
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2302_12519_gb300 import build
    build.build()
    ep.load()


# A chunk of 2 048 rows is cut into 16 shares for a small batch (chunks of 2 048, 1 and 304 rows), into 7 for 64 x 6
# chunks, and stays whole from 2 737 chunks on; one member of each batch is too small for tables.
@pytest.mark.parametrize("sizes", [[(16, 16, 16), (17, 241, 1)], [(20, 20, 11)], [(23, 22, 21)] * 64, [(88, 88, 88)] * 9],
                         ids=["16 shares", "partial chunk", "7 shares", "whole chunks"])
def test_monodomain_members_same_alone_and_in_the_mix(sizes):
    cases = [W.random_case(70 + i, *n, model=W.MONO, mask=np.ones(n[::-1], np.uint8))
             for i, n in enumerate(sizes + [(12, 11, 10)])]
    for c in cases:
        c.stimuli = [W.Stimulus((0, 0, 0), (5, 5, 1), 0.1, 0.1, 0.5)]   # steps 2 and 3
    both = []
    for _ in range(2):
        both.append([ep.sim_from_case(c) for c in cases])
        for i, (s, c) in enumerate(zip(both[-1], cases)):
            v, w, _ = W.random_state(70 + i, c)
            s.set_state(v, w, None, i % 2)   # members on even and on odd steps
    alone, mixed = both
    b = ep.Batch(len(cases))
    for s in mixed:
        b.add(s)
    b.step(2)
    b.step(3)
    for a, m in zip(alone, mixed):
        a.step(5)
        for f in (ep.EP_V, ep.EP_W, ep.EP_TACT):
            np.testing.assert_array_equal(m.read(f), a.read(f))
    b.close()
    for s in alone + mixed:
        s.close()


# Blocks above the 720 thousand voxels up to which they have tables, one full and one with a cavity: the planes of a work
# item change with the schedule (8 to 32 of 40), and with them which voxels lie in items without a hole
@pytest.mark.parametrize("cavity", [False, True])
def test_results_do_not_depend_on_the_planes_of_a_work_item(cavity):
    mask = np.ones((40, 150, 150), np.uint8)
    if cavity:
        mask[18:22, 60:63, 70:90] = 0
    c = W.random_case(81, 150, 150, 40, model=W.MONO, mask=mask)
    v, w, _ = W.random_state(81, c)
    out = []
    for zseg in (None, 8, 16, 32):
        s = ep.sim_from_case(c)
        s.set_state(v, w, None, 0)
        if zseg is None:
            s.step(3)
        else:
            b = ep.Batch(1)
            b.set_schedule(0, zseg, -1)
            b.add(s)
            b.step(3)
            b.close()
        out.append([s.read(f) for f in (ep.EP_V, ep.EP_W, ep.EP_TACT)])
        s.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)

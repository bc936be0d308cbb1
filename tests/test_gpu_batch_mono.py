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

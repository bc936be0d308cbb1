"""Dense blocks at the sizes where the sweep takes another form by its cost, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_2302_12519_gb300 as ep
import workloads as W

pytestmark = pytest.mark.gpu

SWEEPS = 4


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2302_12519_gb300 import build
    build.build()
    ep.load()


# rows to march (Jacobi) and bricks (Chebyshev) above about 320 thousand voxels, a block with holes, bricks to march
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("nx,ny,nz,fill", [(64, 65, 66, 1.0), (73, 75, 74, 1.0), (80, 79, 81, 0.97), (141, 140, 131, 1.0)])
def test_dense_blocks(nx, ny, nz, fill, solver):
    mask = (np.random.default_rng(1).random((nz, ny, nx)) < fill).astype(np.uint8)
    c = W.random_case(21, nx, ny, nz, mask=mask).fibres_as_float32()
    p = c.params
    p.solver, p.max_iter, p.rel_tol, p.check_every = solver, SWEEPS, 0.0, 2
    p.cheb_lmin, p.cheb_lmax = (0.01, 5.5) if solver == 1 else (0.0, 0.0)
    v, w, ve = W.random_state(21, c)
    s, ref = ep.sim_from_case(c), oracle.Sim(c)
    s.set_state(v, w, ve, 0)
    ref.set_state(v, w, ve, 0)
    assert s.step(1, allow_noconv=True).iters == SWEEPS
    ref.step()
    want = ref.state()["ve"]
    # 32 roundings of 2^-24 of 6 max|x| a sweep, and four more of v, the right-hand side and the start
    tol = (32 * 6 * SWEEPS + 4 * 32) * 2.0 ** -24 * max(1.0, float(np.abs(want).max()))
    assert np.abs(s.read(ep.EP_VE) - want).max() <= tol
    s.close()
    ref.close()

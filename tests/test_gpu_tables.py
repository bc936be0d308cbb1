"""The tabulated operator (assembled rows and bricks) and the walk over clear items against the FP64 oracle: a few
capped sweeps or steps from a random state, so that every voxel's value depends on its own entries, at sizes around
the edges of a row CTA (128 rows), a brick (30 x 6 x 8 voxels), a work item (30 x 7 x 32), ragged grids, grids with
holes and thin ones."""
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


def _mask(kind, seed, nx, ny, nz):
    rng = np.random.default_rng(seed)
    if kind == "full":
        return np.ones((nz, ny, nx), np.uint8)
    if kind == "holes":
        return (rng.random((nz, ny, nx)) > 0.03).astype(np.uint8)
    return W.random_mask(rng, nx, ny, nz, 0.8)


def _check(kind, seed, nx, ny, nz, solver, precision):
    c = W.random_case(seed, nx, ny, nz, mask=_mask(kind, seed, nx, ny, nz), precision=precision).fibres_as_float32()
    p = c.params
    p.solver, p.max_iter, p.rel_tol, p.check_every = solver, SWEEPS, 0.0, 2
    p.cheb_lmin, p.cheb_lmax = (0.01, 5.5) if solver == 1 else (0.0, 0.0)
    p.omega = 1.3 if solver == 2 else 0.0
    v, w, ve = W.random_state(seed, c)
    s, ref = ep.sim_from_case(c), oracle.Sim(c)
    s.set_state(v, w, ve, 0)
    ref.set_state(v, w, ve, 0)
    st = s.step(1, allow_noconv=True)
    ref.step()
    assert st.iters == SWEEPS
    want = ref.state()
    # a sweep moves a voxel by omega / D times sums of at most 26 products of coefficients (their sum at most 6 D)
    # and values: 32 roundings of 2^-24 (FP64: 2^-53, but 1/D is stored in FP32) of 6 max|x| a sweep, after the
    # rounding of v, the right-hand side and the start, four more of the same size
    x = max(1.0, float(np.abs(want["ve"]).max()))
    eps = 2.0 ** -24
    tol = (32 * 6 * SWEEPS + 4 * 32) * eps * x if precision == W.FP32 else 6 * SWEEPS * eps * x
    assert np.abs(s.read(ep.EP_VE) - want["ve"]).max() <= tol
    s.close()
    ref.close()


# up to 720 000 tissue voxels: rows.  4 096 is the smallest tabulated handle, 4 095 the largest general one.
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("solver", [0, 1, 2])
@pytest.mark.parametrize("kind,nx,ny,nz", [("full", 16, 16, 16), ("full", 4095, 1, 1), ("holes", 33, 31, 29),
                                           ("blobs", 47, 40, 23), ("full", 2, 64, 65)])
def test_rows(kind, nx, ny, nz, solver, precision):
    _check(kind, 3, nx, ny, nz, solver, precision)


# 37 steps from step 3 (one step to an even one, a graph of 32, four more), a stimulus that starts and ends inside
@pytest.mark.parametrize("diffusion", [0, 1])
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("kind,nx,ny,nz", [("full", 17, 16, 16), ("holes", 33, 23, 19), ("full", 4200, 1, 1)])
def test_monodomain_rows(kind, nx, ny, nz, precision, diffusion):
    c = W.random_case(7, nx, ny, nz, model=W.MONO, mask=_mask(kind, 7, nx, ny, nz),
                      precision=precision).fibres_as_float32()
    c.params.diffusion = diffusion
    c.params.rel_tol = 1e-12 if precision == W.FP64 else 1e-6
    c.stimuli = [W.Stimulus((1, 0, 0), (nx - 1, 5, 5), 0.4, 0.6, 0.5)]
    v, w, _ = W.random_state(7, c)
    s, ref = ep.sim_from_case(c), oracle.Sim(c)
    s.set_state(v, w, None, 3)
    ref.set_state(v, w, None, 3)
    assert s.step(37).step == 40
    for _ in range(37):
        ref.step()
    want = ref.state()
    # 40 roundings of 2^-24 a step (FP64: of 2^-53, and the implicit solves' 1e-12), carried at most exp(37 dt 0.25 / tau_in)
    grow = np.exp(37 * c.params.dt * 0.25 / c.params.tau_in)
    tol = 37 * grow * (40 * 2.0 ** -24 + (1e-6 if diffusion else 0.0)) if precision == W.FP32 else \
        37 * grow * (40 * 2.0 ** -53 + (1e-11 if diffusion else 0.0))
    assert np.abs(s.read(ep.EP_V) - want["v"]).max() <= tol
    assert np.abs(s.read(ep.EP_W) - want["w"]).max() <= tol
    a, b = s.read(ep.EP_TACT), want["tact"]
    assert np.array_equal(a >= 0, b >= 0) and np.abs(a - b).max() <= 100 * tol
    s.close()
    ref.close()


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("kind,nx,ny,nz", [("full", 91, 91, 89), ("holes", 120, 84, 78), ("holes", 31, 161, 151),
                                           ("blobs", 122, 107, 91)])
def test_bricks(kind, nx, ny, nz, solver):
    _check(kind, 5, nx, ny, nz, solver, W.FP32)


# above 720 000 voxels the FP32 monodomain walks; a block is made of clear items (31 x 151 x 155 and 91 x 91 x 89 end
# inside a window, a row band and a plane block), one with a hole of clear and general ones
@pytest.mark.parametrize("diffusion", [0, 1])
@pytest.mark.parametrize("kind,nx,ny,nz", [("full", 91, 91, 89), ("full", 31, 151, 155), ("hole", 120, 85, 78)])
def test_clear_items(kind, nx, ny, nz, diffusion):
    mask = np.ones((nz, ny, nx), np.uint8)
    if kind == "hole":
        mask[40:44, 30:33, 50:60] = 0
    c = W.random_case(9, nx, ny, nz, model=W.MONO, mask=mask).fibres_as_float32()
    c.params.diffusion = diffusion
    v, w, _ = W.random_state(9, c)
    s, ref = ep.sim_from_case(c), oracle.Sim(c)
    s.set_state(v, w, None, 0)
    ref.set_state(v, w, None, 0)
    s.step(3)
    for _ in range(3):
        ref.step()
    want = ref.state()
    grow = np.exp(3 * c.params.dt * 0.25 / c.params.tau_in)
    tol = 3 * grow * (40 * 2.0 ** -24 + (1e-6 if diffusion else 0.0))   # as above
    assert np.abs(s.read(ep.EP_V) - want["v"]).max() <= tol
    assert np.abs(s.read(ep.EP_W) - want["w"]).max() <= tol
    s.close()
    ref.close()


# heart in a torso: rows near the tissue and around holes of the torso, the walk away from them (items of 30 x 7 x 8
# at these sizes, cut by the box)
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("nx,ny,nz,fill", [(64, 47, 53, None), (91, 40, 61, 0.9995), (40, 38, 36, 0.9)])
def test_torso_rows_and_walk(nx, ny, nz, fill, solver):
    z, y, x = np.meshgrid(*[np.arange(n) + 0.5 - n / 2 for n in (nz, ny, nx)], indexing="ij")
    r = np.sqrt(x * x + y * y + z * z)
    c = W.random_case(11, nx, ny, nz, mask=((r < 14) & (r > 7)).astype(np.uint8)).fibres_as_float32()
    c = W.with_torso(c, sig_o=0.8, fill=fill, seed=2)
    p = c.params
    p.solver, p.max_iter, p.rel_tol, p.check_every = solver, SWEEPS, 0.0, 2
    p.cheb_lmin, p.cheb_lmax = (0.01, 6.0) if solver == 1 else (0.0, 0.0)
    v, w, ve = W.random_state(11, c)
    s, ref = ep.sim_from_case(c), oracle.Sim(c)
    s.set_state(v, w, ve, 0)
    ref.set_state(v, w, ve, 0)
    assert s.step(1, allow_noconv=True).iters == SWEEPS
    ref.step()
    want = ref.state()["ve"]
    tol = (32 * 6 * SWEEPS + 4 * 32) * 2.0 ** -24 * max(1.0, float(np.abs(want).max()))   # as for the rows
    assert np.abs(s.read(ep.EP_VE) - want).max() <= tol
    s.close()
    ref.close()


@pytest.mark.parametrize("kind,nx,ny,nz", [("torso", 64, 47, 53), ("full", 91, 91, 89), ("full", 33, 31, 29)])
def test_differences_of_large_values(kind, nx, ny, nz):
    """The residual of a start that is large against its differences (2^14 and 0 to 4 units in the last place) is the
    FP64 operator's on the same start and the same new v: neighbours are subtracted before anything is added."""
    mask = np.ones((nz, ny, nx), np.uint8)
    if kind == "torso":
        z, y, x = np.meshgrid(*[np.arange(n) + 0.5 - n / 2 for n in (nz, ny, nx)], indexing="ij")
        r = np.sqrt(x * x + y * y + z * z)
        mask = ((r < 14) & (r > 7)).astype(np.uint8)
    h = []
    for precision in (W.FP32, W.FP64):
        c = W.random_case(13, nx, ny, nz, mask=mask, precision=precision).fibres_as_float32()
        if kind == "torso":
            c = W.with_torso(c, sig_o=0.8)
        c.params.max_iter, c.params.rel_tol, c.params.check_every = 1, 0.0, 1
        h.append(ep.sim_from_case(c))
    v, w, ve = W.random_state(13, c)
    far = 2.0 ** 14 + 2.0 ** -9 * np.random.default_rng(13).integers(0, 5, ve.size)
    far = np.where(ve != 0.0, far, 0.0)
    h[0].set_state(2.0 ** -10 * v, w, far, 0)
    got = h[0].step(1, allow_noconv=True).rel_res
    b = -h[1].apply_operator(c.params.sig_iL, c.params.sig_iT, h[0].read(ep.EP_V))
    want = np.linalg.norm(b - h[1].apply_elliptic(far)) / np.linalg.norm(b)
    for s in h:
        s.close()
    # the rounding of a residual, as above, is under 32 x 6 of 2^-24 of its terms, in norm far less; sums of values
    # would be off by one unit of 2^14 in every second one, a tenth of the residual
    assert abs(got / want - 1.0) <= 1e-4


def test_tables_give_way_to_a_budget():
    """A batch budget that two handles meet without their tables, but not with them, admits both; they give the
    results of a handle that never had tables to the rounding of the operator's two forms."""
    c = W.random_case(8, 40, 30, 20, mask=np.ones((20, 30, 40), np.uint8))
    hs = [ep.sim_from_case(c, use_torch=False) for _ in range(3)]
    v, w, ve = W.random_state(8, c)
    for h in hs:
        h.set_state(v, w, ve, 0)
    full = hs[0].info().device_bytes
    rows = 112 * c.n_tissue
    b = ep.Batch(2, hbm_budget_bytes=2 * full - rows)
    for h in hs[:2]:
        b.add(h)
    assert sum(h.info().device_bytes for h in hs[:2]) <= 2 * full - rows
    b.step(2)
    hs[2].step(2)
    for h in hs[:2]:
        assert np.abs(h.read(ep.EP_VE) - hs[2].read(ep.EP_VE)).max() <= 1e-5
    b.close()
    for h in hs:
        h.close()

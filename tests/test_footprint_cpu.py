"""The sizes of the operator tables that ep.h states, from ep_footprint's plan on the host."""
import numpy as np
import pytest

import paper_2302_12519_gb300 as ep
import workloads as W


@pytest.fixture(scope="module")
def lib():
    from paper_2302_12519_gb300 import build
    build.build()
    return ep.load()


def _tables(c, torso=None):
    """Table bytes: what the parameters add to the plan of the mask, less the third iterate of an FP32 solve."""
    s = ep.Sim(c.nx, c.ny, c.nz, c.dx, c.model, c.precision, use_torch=False)
    s.set_mask(c.mask_flat())
    if torso is not None:
        s.set_torso(torso, 1.0)
    before = s.footprint()[0]
    s.set_params(c.params)
    after = s.footprint()[0]
    s.close()
    third = 4 * c.n if c.model == W.BI and c.precision == W.FP32 and c.params.solver != 2 else 0
    return after - before - third


# besides the entries a voxel: 8 192 weights, 33 counters of 128 bytes and the sweeps' partial sums
EXTRA = 8 * 8192 + 33 * 128 + 8 * 8 * 4096 + 16


@pytest.mark.parametrize("model,precision,solver,per", [(W.BI, W.FP32, 0, 112), (W.BI, W.FP32, 2, 112), (W.MONO, W.FP32, 0, 112),
                                                        (W.BI, W.FP64, 1, 224), (W.MONO, W.FP64, 0, 224)])
def test_row_tables(lib, model, precision, solver, per):
    c = W.random_case(3, 40, 41, 43, model=model, precision=precision, mask=np.ones((43, 41, 40), np.uint8))
    c.params.solver = solver
    assert 0 <= _tables(c) - per * c.n_tissue <= EXTRA


@pytest.mark.parametrize("kind", ["box", "heart"])
def test_brick_tables(lib, kind):
    c = W.random_case(3, 91, 91, 89, mask=np.ones((89, 91, 91), np.uint8)) if kind == "box" else W.config2(n=160)
    c.params.solver = 1 if kind == "box" else 0   # the Jacobi sweeps of a box that large take the march
    assert 43.0 < _tables(c) / c.n_tissue < 50.0


def test_no_tables(lib):
    for c in (W.random_case(3, 16, 16, 15, mask=np.ones((15, 16, 16), np.uint8)),
              W.random_case(3, 91, 91, 89, model=W.MONO, mask=np.ones((89, 91, 91), np.uint8))):
        assert _tables(c) == 0


@pytest.mark.parametrize("n,fill,jacobi,chebyshev", [(64, 1.0, 112, 112), (74, 1.0, 0, 45), (88, 1.0, 0, 45), (150, 1.0, 0, 0),
                                                     (80, 0.97, 0, 45)])
def test_form_of_a_dense_block(lib, n, fill, jacobi, chebyshev):
    """Bytes a tissue voxel: rows, none (the march), bricks."""
    mask = (np.random.default_rng(1).random((n, n, n)) < fill).astype(np.uint8)
    for solver, per in ((0, jacobi), (1, chebyshev)):
        c = W.random_case(3, n, n, n, mask=mask)
        c.params.solver = solver
        assert abs(_tables(c) / c.n_tissue - per) <= (6 if per else 0)


@pytest.mark.parametrize("case,per", [(W.config1(), 112), (W.config2(n=144), 112), (W.config2(n=176), 45), (W.sampled_shell(np.random.default_rng(0), 204, 1, "s"), 45)],
                         ids=["shell128", "heart144", "heart176", "shell204"])
def test_form_of_shells_and_hearts(lib, case, per):
    for solver in (0, 1):
        case.params.solver = solver
        assert abs(_tables(case) / case.n_tissue - per) <= 5


def test_torso_tables(lib):
    """Rows for the tissue and the torso voxels at it, 4 bytes for every voxel of the grid, and the work items."""
    c = W.config2(n=64)
    torso = (c.mask == 0).astype(np.uint8)
    pad = np.pad(c.mask > 0, 1)
    near = np.zeros_like(pad)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                near |= np.roll(pad, (dz, dy, dx), (0, 1, 2))
    rows = int(near[1:-1, 1:-1, 1:-1].sum())
    assert 0 <= _tables(c, torso) - 112 * rows - 4 * c.n <= EXTRA + 16 * c.n // (30 * 7 * 8) * 4

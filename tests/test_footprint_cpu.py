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
    assert 43.0 < _tables(c) / c.n_tissue < 50.0


def test_no_tables(lib):
    for c in (W.random_case(3, 16, 16, 15, mask=np.ones((15, 16, 16), np.uint8)),
              W.random_case(3, 91, 91, 89, model=W.MONO, mask=np.ones((89, 91, 91), np.uint8))):
        assert _tables(c) == 0


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

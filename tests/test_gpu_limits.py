"""Where memory or the stream sets a limit: budgets and allocators that hold a handle's fields but not its operator
tables, a handle held by two batches, streams that cannot be captured.  None of it faults the GPU: budgets and
allocators refuse on the host."""
import numpy as np
import pytest

import oracle
import paper_2302_12519_gb300 as ep
import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = (ep.EP_V, ep.EP_W, ep.EP_VE, ep.EP_TACT)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2302_12519_gb300 import build
    build.build()
    ep.load()


@pytest.mark.parametrize("change", ["budget", "work items"])
def test_a_handle_in_two_batches(change):
    """A handle that another batch strips of its operator tables (a budget that only bare handles meet), or gives other
    work items, is stepped right by the batch that held it before, whose lists were built on what it had."""
    tabulated = change == "budget"
    nx, ny, nz = (40, 30, 20) if tabulated else (12, 10, 30)   # 3 600 voxels have no tables
    cases = [W.random_case(14 + i, nx - i, ny, nz, mask=np.ones((nz, ny, nx - i), np.uint8)) for i in range(2)]
    for c in cases:
        c.params.max_iter, c.params.rel_tol, c.params.check_every = 4, 0.0, 2
    hs = [[ep.sim_from_case(c) for c in cases] for _ in range(2)]
    for pair in hs:
        for i, (h, c) in enumerate(zip(pair, cases)):
            h.set_state(*W.random_state(14 + i, c), 0)
    (a, other), alone = hs[0], hs[1][0]
    first = ep.Batch(1)
    first.set_schedule(0, 64, 0)
    first.add(a)
    first.step(2, allow_noconv=True)
    budget = 0
    if tabulated:   # room for the other handle's tables at most
        rows = 112 * cases[0].n_tissue
        budget = a.info().device_bytes + other.info().device_bytes - rows
    second = ep.Batch(2, hbm_budget_bytes=budget)
    second.set_schedule(0, 64 if tabulated else 8, 0)
    second.add(other)
    held = a.info().device_bytes
    second.add(a)
    assert (a.info().device_bytes < held) == tabulated
    first.step(2, allow_noconv=True)
    second.step(1, allow_noconv=True)
    alone.step(5, allow_noconv=True)
    # five steps of four sweeps over the operator's other form: 32 roundings of 2^-24 of 6 max|x| a sweep, four more a
    # step for v and the right-hand side, carried at most exp(5 dt 0.25 / tau_in)
    p = cases[0].params
    tol = 5 * (32 * 6 * 4 + 4 * 32) * 2.0 ** -24 * np.exp(5 * p.dt * 0.25 / p.tau_in)
    for f in FIELDS[:3]:
        assert np.abs(a.read(f) - alone.read(f)).max() <= tol * max(1.0, float(np.abs(alone.read(f)).max()))
    first.close()
    second.close()
    for h in hs[0] + hs[1]:
        h.close()


@pytest.mark.parametrize("model,precision", [(W.BI, W.FP64), (W.MONO, W.FP64), (W.BI, W.FP32)])
def test_an_allocator_that_aligns_to_16_bytes(model, precision):
    """Every block lies 16 bytes past a 32-byte boundary: the results are those of well aligned memory, bit for bit."""
    alloc, free = ep.torch_allocator()
    c = W.random_case(33, 17, 16, 16, model=model, mask=np.ones((16, 16, 17), np.uint8), precision=precision)
    c.params.max_iter, c.params.rel_tol, c.params.check_every = 5, 0.0, 2
    v, w, ve = W.random_state(33, c)
    out = []
    for pair in ((alloc, free), (lambda n: alloc(n + 16) + 16, lambda p: free(p - 16))):
        s = ep.sim_from_case(c, allocator=pair)
        s.set_state(v, w, ve, 0)
        s.step(2, allow_noconv=True)
        resident = s.info().device_bytes
        assert resident == s.footprint()[0]
        out.append([s.read(f) for f in FIELDS])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


CUDA_STREAM_LEGACY = 1   # cudaStreamLegacy: the default stream, which cannot be captured


# 70 steps: two graphs of 32 and six single launches
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
def test_monodomain_steps_on_a_stream_that_cannot_be_captured(precision):
    c = W.random_case(31, 17, 16, 16, model=W.MONO, mask=np.ones((16, 16, 17), np.uint8), precision=precision)
    v, w, _ = W.random_state(31, c)
    out = []
    for stream in (None, CUDA_STREAM_LEGACY):
        s = ep.Sim(c.nx, c.ny, c.nz, c.dx, ep.EP_MONO, precision, use_torch=False, stream=stream)
        s.set_mask(c.mask_flat())
        s.set_fibres(c.fib_flat())
        s.set_params(c.params)
        s.set_state(v, w, None, 0)
        assert s.step(70).step == 70
        out.append([s.read(f) for f in FIELDS])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def _shell(seed):
    """Few tissue voxels in a large box: its tables (112 bytes a tissue voxel) are less than the set-up's staging."""
    c = W.sampled_shell(np.random.default_rng(seed), 48, 10, f"shell{seed}")
    c.params.max_iter, c.params.rel_tol = 50, 0.0
    return c, ep.sim_from_case(c, use_torch=False)


def _sizes():
    """Device bytes of such a handle and the peak of its set-up, with tables and without."""
    c, s = _shell(0)
    resident, peak = s.footprint()
    s.close()
    tables = 112 * c.n_tissue
    assert c.n_tissue >= 4096 and peak - resident > tables   # so that one handle alone fits every budget below
    return resident, peak, resident - tables, peak - tables


SLACK = 1 << 17   # the Chebyshev weights, counters and partial sums that belong to the tables


# What two requests need at once: the second without its tables; both without; the first a result not yet collected.
@pytest.mark.parametrize("who", ["second", "both", "result"])
def test_server_gives_tables_up_to_admit(who):
    resident, peak, bare, bare_peak = _sizes()
    budget = (resident if who == "second" else bare) + bare_peak + SLACK
    assert peak <= budget < resident + peak
    srv = ep.Server(max_slots=4, chunk_steps=2, hbm_budget_bytes=budget)
    first = srv.submit(_shell(0)[1], 2 if who == "result" else 400)
    if who == "result":
        srv.drain(timeout_s=60)
    second = srv.submit(_shell(0)[1], 2)
    srv.drain(timeout_s=60)   # EP_EBUSY if the second request waits for the first one's memory
    got = {r.id: (r, s) for r, s in srv.collect(max_results=4)}
    assert {first, second} == set(got)
    for r, s in got.values():
        assert r.status in (ep.EP_OK, ep.EP_ENOCONV) and r.device_bytes == s.info().device_bytes
    if who != "result":
        assert got[second][0].t_admit_s < got[first][0].t_done_s
    assert (got[first][0].device_bytes < resident) == (who != "second") and got[second][0].device_bytes < resident
    assert srv.stats().hbm_peak <= budget and srv.stats().hbm_in_use == 0
    srv.close()
    if who != "both":
        return
    c, alone = _shell(0)   # both ran on without tables: two steps against a handle that has them
    alone.step(2, allow_noconv=True)
    # 50 sweeps a step, 32 roundings of 2^-24 of 6 max|x| a sweep and four more a step for v and the right-hand side
    tol = 2 * (32 * 6 * 50 + 4 * 32) * 2.0 ** -24
    for f in FIELDS[:3]:
        assert np.abs(got[second][1].read(f) - alone.read(f)).max() <= tol * max(1.0, float(np.abs(alone.read(f)).max()))
    alone.close()


def test_server_takes_a_set_up_handle_without_its_tables():
    """A handle that comes with its tables, for a budget that it meets without them."""
    resident, _, bare, _ = _sizes()
    s = _shell(0)[1]
    assert s.info().device_bytes == resident
    srv = ep.Server(max_slots=1, hbm_budget_bytes=bare + SLACK)
    srv.submit(s, 2)
    srv.drain(timeout_s=60)
    (r, s), = srv.collect()
    assert r.status in (ep.EP_OK, ep.EP_ENOCONV) and r.steps_done == 2 and r.device_bytes <= bare + SLACK
    s.close()
    srv.close()


def test_server_leaves_a_rejected_handle_its_tables():
    _, _, bare, bare_peak = _sizes()
    fresh, ready = _shell(0)[1], _shell(0)[1]
    held = ready.info().device_bytes
    plan = fresh.footprint()
    srv = ep.Server(max_slots=2, hbm_budget_bytes=bare - SLACK)
    ids = [srv.submit(fresh, 2), srv.submit(ready, 2)]
    srv.drain(timeout_s=60)
    got = {r.id: (r, s) for r, s in srv.collect()}
    assert all(got[i][0].status == ep.EP_EREJECTED for i in ids)
    assert got[ids[0]][1].footprint() == plan and got[ids[1]][1].info().device_bytes == held
    srv.close()


class CappedAllocator:
    """torch's caching allocator behind the dev_alloc / dev_free hooks, up to `cap` bytes at a time."""

    def __init__(self, cap):
        self.alloc, self.free = ep.torch_allocator()
        self.cap, self.size = cap, {}

    def pair(self):
        def alloc(nbytes):
            if sum(self.size.values()) + nbytes > self.cap:
                return 0
            p = self.alloc(nbytes)
            self.size[p] = nbytes
            return p

        def free(ptr):
            del self.size[ptr]
            self.free(ptr)

        return alloc, free


# the last row: a colour pass over rows, bricks (737 thousand voxels), rows and the torso's walk
@pytest.mark.parametrize("kind,model,precision,solver", [("box", W.BI, W.FP32, 1), ("box", W.BI, W.FP64, 0),
                                                         ("box", W.MONO, W.FP32, 0), ("box", W.MONO, W.FP64, 0),
                                                         ("box", W.BI, W.FP32, 2), ("big", W.BI, W.FP32, 1),
                                                         ("torso", W.BI, W.FP32, 1)])
def test_tables_that_do_not_fit_are_left_out(kind, model, precision, solver):
    """Memory for a handle's fields and staging but not its tables: it steps without them, to the rounding of the
    operator's two forms of the oracle; and after an attempt that had no room at all, a later one gets its tables."""
    nx, ny, nz = {"box": (23, 20, 19), "big": (91, 91, 89), "torso": (47, 40, 41)}[kind]
    mask = np.ones((nz, ny, nx), np.uint8)
    if kind == "torso":
        z, y, x = np.meshgrid(*[np.arange(n) + 0.5 - n / 2 for n in (nz, ny, nx)], indexing="ij")
        r = np.sqrt(x * x + y * y + z * z)
        mask = ((r < 14) & (r > 7)).astype(np.uint8)
    c = W.random_case(35, nx, ny, nz, model=model, mask=mask, precision=precision).fibres_as_float32()
    if kind == "torso":
        c = W.with_torso(c, sig_o=0.8)
    p = c.params
    p.solver, p.max_iter, p.rel_tol, p.check_every = solver, 4, 0.0, 2
    p.cheb_lmin, p.cheb_lmax = (0.01, 6.0) if solver == 1 else (0.0, 0.0)
    p.omega = 1.3 if solver == 2 else 0.0
    probe = ep.sim_from_case(c)
    full = probe.footprint()
    probe.close()
    mem = CappedAllocator(full[1] // 8)
    s = ep.sim_from_case(c, allocator=mem.pair())
    with pytest.raises(ep.EPError) as e:
        s.info()
    assert e.value.status == ep.EP_ENOMEM and not mem.size
    assert s.footprint() == full
    mem.cap = full[1] - 1   # one byte short of the tables
    held = s.info().device_bytes
    assert held == sum(mem.size.values()) < full[0]
    v, w, ve = W.random_state(35, c)
    ref = oracle.Sim(c)
    s.set_state(v, w, ve, 0)
    ref.set_state(v, w, ve, 0)
    s.step(1, allow_noconv=True)
    ref.step()
    want = ref.state()
    # four sweeps of 32 roundings of 2^-24 (FP64: 1/D is stored in FP32) of 6 max|x|, and v and the right-hand side
    for f, k in ((ep.EP_V, "v"), (ep.EP_W, "w")) + (((ep.EP_VE, "ve"),) if model == W.BI else ()):
        x = max(1.0, float(np.abs(want[k]).max()))
        tol = (32 * 6 * 4 + 4 * 32) * 2.0 ** -24 * x if precision == W.FP32 else 6 * 4 * 2.0 ** -24 * x
        assert np.abs(s.read(f) - want[k]).max() <= tol
    s.close()
    ref.close()
    assert not mem.size
    mem.cap = full[1]
    s = ep.sim_from_case(c, allocator=mem.pair())
    mem.cap = full[1] // 8
    with pytest.raises(ep.EPError):
        s.info()
    mem.cap = full[1]
    assert s.info().device_bytes == full[0]
    s.close()

"""The bulk-copy sweep's device-side failure path, exercised without a fault.

Every mbarrier wait of the bulk-copy sweep is bounded; a wait that runs out
sets the step control's error word, the CTA's producer waits (bounded) for
its own copies in flight, and the call returns LBMBT_EDEVICE.  The test-only
option LBMBT_OPT_TEST_WAIT_NS makes each consumer warp first wait, with a
short limit, on a shared-memory barrier that nothing completes, so the wait
runs out as one for a lost copy would.  The grid is tiny (one unit per CTA),
so the producer never waits for a stage to be released.  The next run on the
same context, with the option off, matches the oracle.
"""
import math
import threading
import time

import numpy as np
import pytest

import oracle
from paper_1907_00908_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    from paper_1907_00908_gb300 import lbmbt
    lbmbt.lib()
    return lbmbt


@pytest.mark.parametrize("n_steps", [4, 20])   # 20: the steps replay as a captured graph
def test_wait_timeout_reports_edevice_and_the_context_recovers(lb, n_steps):
    rng = np.random.default_rng(9)
    geom = synth.Geometry(rng.integers(0, 2, size=(2, 4, 16)).astype(np.int32), np.array([0, 1], np.uint8), 0.5)
    dt = 0.02
    gG = [0.05, 0.0, 0.03]
    f = np.ones(n_steps)
    D, T2, kap = [2.0, 1.0], [80.0, 50.0], 0.04
    s = lb.Solver(0)
    s.set_option(lb.OPT_KERNEL, 2)
    s.set_geometry(geom.labels, geom.phase_of_label, geom.dx)
    s.set_phases(D, T2)
    s.set_permeability(kap)
    s.set_sequence(dt, f, gG)
    assert s.get_option(lb.OPT_TEST_WAIT_NS) == 0          # off unless a test sets it
    s.set_option(lb.OPT_TEST_WAIT_NS, 1_000_000)           # 1 ms
    t0 = time.perf_counter()
    with pytest.raises(lb.LbmbtError) as e:
        s.run()
    assert e.value.code == -6 and "timed out" in str(e.value)
    assert time.perf_counter() - t0 < 5.0
    s.set_option(lb.OPT_TEST_WAIT_NS, 0)
    fld = torch.zeros(geom.n_sites, dtype=torch.complex64, device="cuda")
    r = s.run(field=fld)
    torch.cuda.synchronize()
    assert s.get_option(lb.OPT_KERNEL_USED) == 2
    s.close()
    o = oracle.run(geom.labels, geom.dx, geom.phase_of_label, (0, 0, 0), D, T2, kap, dt, f, gG, want_field=True)
    assert abs(r["S"] - o["S"]) <= 1e-5 * o["S"]
    err = np.abs(fld.cpu().numpy().reshape(geom.labels.shape) - o["field"]).max() / np.abs(o["field"]).max()
    assert err < 1e-4 and math.isfinite(r["S"])


def test_test_wait_option_bounds(lb):
    s = lb.Solver(0)
    for bad in (-1, 1_000_000_001):
        with pytest.raises(lb.LbmbtError):
            s.set_option(lb.OPT_TEST_WAIT_NS, bad)
    s.close()


def _times_out_and_recovers(lb, s, call, geom, bc, D, T2, kap, dt, f, gG):
    """`call` fails with EDEVICE while the first wait runs out; then the same
    context runs as the oracle does."""
    s.set_option(lb.OPT_TEST_WAIT_NS, 1_000_000)           # 1 ms
    t0 = time.perf_counter()
    with pytest.raises(lb.LbmbtError) as e:
        call()
    assert e.value.code == -6 and "timed out" in str(e.value)
    assert time.perf_counter() - t0 < 5.0
    s.set_option(lb.OPT_TEST_WAIT_NS, 0)
    fld = torch.zeros(geom.n_sites, dtype=torch.complex64, device="cuda")
    r = s.run(field=fld)
    torch.cuda.synchronize()
    o = oracle.run(geom.labels, geom.dx, geom.phase_of_label, bc, D, T2, kap, dt, f, gG, want_field=True,
                   lattice="D2Q5" if s.get_option(lb.OPT_LATTICE) else "D3Q7")
    assert abs(r["S"] - o["S"]) <= 1e-5 * o["S"]
    err = np.abs(fld.cpu().numpy().reshape(geom.labels.shape) - o["field"]).max() / np.abs(o["field"]).max()
    assert err < 1e-4 and math.isfinite(r["S"])


def _setup(lb, shape, n_steps, lattice=0):
    rng = np.random.default_rng(9)
    geom = synth.Geometry(rng.integers(0, 2, size=shape).astype(np.int32), np.array([0, 1], np.uint8), 0.5)
    dt, gG, f, D, T2, kap = 0.02, [0.05, 0.0, 0.0], np.ones(n_steps), [2.0, 1.0], [80.0, 50.0], 0.04
    s = lb.Solver(0)
    s.set_option(lb.OPT_LATTICE, lattice)
    s.set_geometry(geom.labels, geom.phase_of_label, geom.dx)
    s.set_phases(D, T2)
    s.set_permeability(kap)
    s.set_sequence(dt, f, gG)
    return s, (geom, (0, 0, 0), D, T2, kap, dt, f, gG)


# one item and several, two steps and one more, a captured graph, sums in the kernel
# (series) after the waits ran out
@pytest.mark.parametrize("shape", [(4, 6, 18), (40, 21, 37)])
@pytest.mark.parametrize("n_steps,series", [(2, False), (5, False), (20, False), (5, True)])
def test_two_step_sweep_wait_timeout(lb, shape, n_steps, series):
    s, job = _setup(lb, shape, n_steps)
    s.set_option(lb.OPT_MULTI_STEP, 2)
    _times_out_and_recovers(lb, s, lambda: s.run(series=series), *job)
    assert s.get_option(lb.OPT_MULTI_STEP_USED) == 2
    s.close()


# blocks in y and z, a few blocks, 2-D blocks and strips
@pytest.mark.parametrize("shape,lattice", [((24, 31, 40), 0), ((4, 9, 5), 0), ((1, 120, 130), 1), ((1, 600, 900), 1)])
@pytest.mark.parametrize("n_steps,series", [(2, False), (25, False), (5, True)])
def test_resident_sweep_wait_timeout(lb, shape, lattice, n_steps, series):
    s, job = _setup(lb, shape, n_steps, lattice)
    s.set_option(lb.OPT_MULTI_STEP, 3)
    _times_out_and_recovers(lb, s, lambda: s.run(series=series), *job)
    assert s.get_option(lb.OPT_MULTI_STEP_USED) == 3
    s.close()


def test_resident_gradient_wait_timeout(lb):
    s, job = _setup(lb, (20, 24, 32), 11)
    geom, gG, kap = job[0], job[7], job[4]
    m = lb.Solver.members([gG], 0, kap)
    _times_out_and_recovers(lb, s, lambda: s.grad_batch(m, checkpoint_every=4), *job)
    after = s.grad_batch(m, checkpoint_every=4)
    s.close()
    s, _ = _setup(lb, (20, 24, 32), 11)
    fresh = s.grad_batch(m, checkpoint_every=4)
    s.close()
    for key in ("S", "dD", "dT2", "dkappa"):
        np.testing.assert_array_equal(after[key], fresh[key])


# the shared memory that a kernel may have is the kernel's, not the context's
@pytest.mark.parametrize("kernel", [2, 0])
def test_a_context_runs_on_after_another_one_with_smaller_blocks_was_prepared(lb, kernel):
    s, job = _setup(lb, (24, 40, 64), 6)
    s.set_option(lb.OPT_KERNEL, kernel)
    s.prepare()
    s.advance(2)
    other, _ = _setup(lb, (2, 2, 16), 6)
    other.set_option(lb.OPT_KERNEL, kernel)
    other.prepare()
    other.advance(2)
    s.advance(4)
    z = s.run()["Z"]
    other.close()
    s.close()
    s, job = _setup(lb, (24, 40, 64), 6)
    s.set_option(lb.OPT_KERNEL, kernel)
    assert s.run()["Z"] == z
    s.close()


KINDS = {"resident": ((9, 31, 20), 0, 3), "strip": ((1, 300, 1300), 1, 3), "links": ((12, 10, 9), 0, 3),
         "resident series": ((9, 31, 20), 0, 3), "two-step": ((40, 21, 37), 0, 2), "gradient": ((20, 24, 32), 0, 0),
         "bulk-copy": ((20, 24, 32), 0, 1), "bulk-copy gradient": ((20, 24, 32), 0, 1)}


def _with_one_failure(lb, kind, fail_at):
    """(first call, second call, allocations to come): the first one's `fail_at`-th allocation
    fails; None where it said ENOMEM."""
    shape, lattice, multi = KINDS[kind]
    s, job = _setup(lb, shape, 4, lattice)
    geom, kap, f, gG = job[0], job[4], job[6], job[7]
    s.set_option(lb.OPT_MULTI_STEP, multi)
    if kind == "links":
        s.set_link_distances(np.random.default_rng(5).uniform(0.1, 0.9, size=(6, *shape)).astype(np.float32))
    m = lb.Solver.members([gG, (0.0, 0.1, 0.0)], 0, kap)
    fields = [torch.zeros(geom.n_sites, dtype=torch.complex64, device="cuda") for _ in range(2)]

    def call():
        if "gradient" in kind:
            r = s.grad_batch(m, checkpoint_every=1)
            return [r["dD"], r["dT2"], r["dkappa"]], np.asarray(r["Z"])
        r = s.run_batch(m, waveforms=[f * 0.5, None], fields=fields, series="series" in kind)
        torch.cuda.synchronize()
        return [v.cpu().numpy() for v in fields], np.asarray(r["Z"])

    first = None
    s.set_option(lb.OPT_TEST_FAIL_ALLOC, fail_at)
    try:
        first = call()
    except lb.LbmbtError as e:
        assert e.code == -2
    left = s.get_option(lb.OPT_TEST_FAIL_ALLOC)
    s.set_option(lb.OPT_TEST_FAIL_ALLOC, 0)
    again = call()
    s.close()
    return first, again, left


# every allocation of a first call fails in turn: the call does without or says
# ENOMEM, and the next call on the context gives what a fresh context gives
@pytest.mark.parametrize("kind", list(KINDS))
def test_each_allocation_may_fail(lb, kind):
    want, _, _ = _with_one_failure(lb, kind, 0)
    tol = 2.0 ** -22 * np.prod(KINDS[kind][0])   # where memory is short the signal may be summed in other groups
    for n in range(1, 60):
        first, again, left = _with_one_failure(lb, kind, n)
        for got in (first, again):
            if got is None:
                continue
            for a, b in zip(got[0], want[0]):
                np.testing.assert_allclose(a, b, rtol=1e-6 if "gradient" in kind else 0, atol=0)
            assert np.abs(got[1] - want[1]).max() <= tol
        if left:
            break
    assert left and n > 8      # the last one came after the last allocation


# what a multi-step sweep needs besides is no reason to refuse a call that the one-step
# sweeps can do
@pytest.mark.parametrize("kind", ["resident", "strip", "links", "two-step", "resident series"])
def test_a_multi_step_run_falls_back_where_memory_is_short(lb, kind):
    n = 1
    while True:
        first, _, left = _with_one_failure(lb, kind, n)
        assert first is not None, n
        if left:
            return
        n += 1


def test_a_resident_gradient_falls_back_where_memory_is_short(lb):
    refused = []
    for kind in ("gradient", "bulk-copy gradient"):
        n, left, k = 1, 0, 0
        while not left:
            first, _, left = _with_one_failure(lb, kind, n)
            k += first is None
            n += 1
        refused.append(k)
    assert refused[0] == refused[1]


def test_resident_stamps_start_over_when_used_up(lb):
    s, job = _setup(lb, (24, 31, 40), 25)
    geom = job[0]
    out = []
    for stamp in (None, 2 ** 32 - 1, 2 ** 32 - 30, None):
        if stamp:
            s.set_option(lb.OPT_TEST_STAMP, stamp)
        fld = torch.zeros(geom.n_sites, dtype=torch.complex64, device="cuda")
        s.run(field=fld)
        torch.cuda.synchronize()
        out.append(fld.cpu().numpy())
        assert s.get_option(lb.OPT_TEST_STAMP) == {0: 26, 1: 26, 2: 2 ** 32 - 5, 3: 26}[len(out) - 1]
    s.close()
    for v in out[1:]:
        np.testing.assert_array_equal(out[0], v)


# a launch takes 32768 steps at most, 4096 with a series
@pytest.mark.parametrize("n_steps,series", [(32768 + 3, False), (2 * 4096 + 1, True)])
def test_resident_run_of_several_launches(lb, n_steps, series):
    out = []
    for multi in (0, 1):
        s, job = _setup(lb, (6, 9, 10), n_steps)
        geom = job[0]
        s.set_sequence(0.02, 1e-3 * np.cos(np.arange(n_steps) * 0.01), [0.05, 0.0, 0.0])
        s.set_phases([2.0, 1.0], [2e4, 2e4])
        s.set_option(lb.OPT_MULTI_STEP, multi)
        fld = torch.zeros(geom.n_sites, dtype=torch.complex64, device="cuda")
        r = s.run(field=fld, series=series)
        torch.cuda.synchronize()
        assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi else 3)
        s.close()
        out.append((fld.cpu().numpy(), r))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][0]).max() > 0.1
    if series:
        assert np.abs(out[0][1]["series"] - out[1][1]["series"]).max() <= 2.0 ** -22 * geom.n_sites


def test_contexts_on_threads_with_blocks_of_different_size(lb):
    shapes = [(20, 24, 32), (40, 48, 48), (7, 5, 16), (60, 57, 57)]
    fail = []

    def work(i):
        try:
            s, job = _setup(lb, shapes[i], 4)
            s.set_option(lb.OPT_MULTI_STEP, 3)
            z = {s.run()["Z"] for _ in range(60)} | {s.grad(checkpoint_every=2)["Z"] for _ in range(10)}
            s.close()
            if len({complex(round(v.real, 6), round(v.imag, 6)) for v in z}) != 1:
                fail.append((i, z))
        except lb.LbmbtError as e:
            fail.append((i, e))

    th = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not fail, fail


# one lost copy in the first sweep; step words written after it where the kept segments
# (7 of 14, 5 of 6, all) start and where segments are recomputed
@pytest.mark.parametrize("every", [3, 7, 40])
def test_gradient_reports_a_time_out_of_its_first_sweep(lb, every):
    s, job = _setup(lb, (4, 6, 16), 40)
    s.set_option(lb.OPT_KERNEL, 2)
    s.set_option(lb.OPT_MULTI_STEP, 1)
    want = s.grad(checkpoint_every=every)
    s.set_option(lb.OPT_TEST_WAIT_SWEEPS, 1)
    s.set_option(lb.OPT_TEST_WAIT_NS, 1_000_000)
    with pytest.raises(lb.LbmbtError) as e:
        s.grad(checkpoint_every=every)
    assert e.value.code == -6 and "timed out" in str(e.value)
    assert s.get_option(lb.OPT_TEST_WAIT_NS) == 0
    again = s.grad(checkpoint_every=every)
    s.close()
    assert again["Z"] == want["Z"] and np.array_equal(again["dD"], want["dD"])


def test_a_closed_context_holds_no_memory(lb):
    def job():
        s, job = _setup(lb, (4, 4, 4), 20000)
        waves = [np.full(20000 - i, 1e-3) for i in range(64)]
        s.run_batch(lb.Solver.members([job[7]] * 64, 0, job[4]), waveforms=waves)
        s.close()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    first = job()
    last = [job() for _ in range(6)][-1]
    assert first - last < 16 << 20      # the 64 waveforms and their integrals take 15 MB a context


@pytest.mark.parametrize("kind", ["time-out", "memory", "none"])
def test_nothing_is_prepared_after_a_gradient_however_it_ended(lb, kind):
    s, job = _setup(lb, (20, 24, 32), 11)
    s.set_option(lb.OPT_TEST_WAIT_NS, 1_000_000 if kind == "time-out" else 0)
    s.set_option(lb.OPT_TEST_FAIL_ALLOC, 14 if kind == "memory" else 0)   # after the forward pass's set-up
    if kind == "none":
        s.grad(checkpoint_every=4)
    else:
        with pytest.raises(lb.LbmbtError) as e:
            s.grad(checkpoint_every=4)
        assert e.value.code == (-6 if kind == "time-out" else -2)
    s.set_option(lb.OPT_TEST_FAIL_ALLOC, 0)
    with pytest.raises(lb.LbmbtError) as e:
        s.advance(1)
    assert e.value.code == -7
    s.close()

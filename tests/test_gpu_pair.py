"""The two-step sweep (LBMBT_OPT_MULTI_STEP = 2) against the one-step register
sweep: the same bits in the field; the signal is summed from the same FP32
thread sums as the one-step sweep that the grid would take otherwise, which
for an nx not a multiple of 16 is the register sweep (FP64 rounding only, 1e-13
of the sum of |M|), else the bulk-copy one (two or three sites a thread: 2^-22
of the sum of |M|); the series within that."""
import math

import numpy as np
import pytest

from paper_1907_00908_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
INF = math.inf


@pytest.fixture(scope="module")
def lb():
    from paper_1907_00908_gb300 import lbmbt
    lbmbt.lib()
    return lbmbt


def _geom(shape, seed, n_labels=3):
    rng = np.random.default_rng(seed)
    coarse = rng.integers(0, n_labels, size=[(n + 2) // 3 for n in shape])
    lab = np.kron(coarse, np.ones((3, 3, 3), int))[:shape[0], :shape[1], :shape[2]]
    return synth.Geometry(np.ascontiguousarray(lab, np.int32), np.arange(n_labels).astype(np.uint8) % 3, 0.5)


def _solver(lb, kernel, geoms, bc, gG, f, kap=0.03):
    s = lb.Solver(0)
    s.set_option(lb.OPT_KERNEL, kernel)
    s.set_option(lb.OPT_MULTI_STEP, 2)
    for i, g in enumerate(geoms):
        (s.add_geometry if i else s.set_geometry)(g.labels, g.phase_of_label, g.dx, bc)
    s.set_phases([2.0, 1.0, 1.5], [80.0, 50.0, INF])
    s.set_permeability(kap)
    s.set_sequence(0.01, f, gG)
    return s


def _wave(kind, n):
    if kind == "pgse":
        f = np.zeros(n)
        f[:max(1, n // 3)] = 1.0
        f[n - max(1, n // 3):] = -1.0
        return f
    return np.cos(np.arange(n) * 0.7)


# tile edges and remainders: one column, one tile, several ragged tiles; the
# smallest nz; faces of every kind
CASES = [
    ((4, 1, 1), (0, 0, 0), (0.3, 0.2, 0.1), "pgse", 7),
    ((4, 5, 3), (0, 0, 0), (0.0, 0.2, 0.4), "pgse", 2),
    ((5, 2, 40), (0, 0, 0), (0.3, 0.0, 0.1), "cos", 9),
    ((37, 23, 31), (0, 0, 0), (0.2, 0.1, -0.3), "pgse", 18),
    ((20, 34, 70), (1, 0, 0), (0.4, 0.0, 0.0), "pgse", 16),
    ((21, 33, 17), (1, 1, 1), (0.0, 0.3, 0.0), "pgse", 33),
    ((40, 12, 64), (1, 1, 1), (0.0, 0.0, 0.5), "cos", 8),
    ((33, 40, 35), (0, 1, 1), (0.3, 0.0, 0.0), "cos", 21),
    ((64, 64, 96), (0, 0, 0), (0.0, 0.0, 0.0), "pgse", 5),
    ((150, 18, 48), (0, 0, 1), (0.2, -0.1, 0.0), "pgse", 34),
]


@pytest.mark.parametrize("shape,bc,gG,wave,n", CASES)
@pytest.mark.parametrize("kap", [0.03, 0.0, INF])
def test_two_step_sweep_gives_the_one_step_bits(lb, shape, bc, gG, wave, n, kap):
    g = _geom(shape, sum(shape))
    f = _wave(wave, n)
    out = []
    for kernel in (0, 1):
        with _solver(lb, kernel, [g], bc, gG, f, kap) as s:
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            r = s.run(field=fld, series=True)
            q = s.run(field=fld)
            torch.cuda.synchronize()
            used = 2 if kernel == 0 and min(shape) >= 4 else 1
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == used
            out.append((fld.cpu().numpy(), r, q))
    assert np.array_equal(out[0][0], out[1][0])
    tol = (1e-13 if shape[2] % 16 else 2.0 ** -22) * np.abs(out[0][0]).sum() + 1e-30
    assert abs(out[0][2]["Z"] - out[1][2]["Z"]) <= tol
    assert out[0][1]["Z"] == out[0][2]["Z"]
    assert np.abs(out[0][1]["series"] - out[1][1]["series"]).max() <= 2.0 ** -22 * g.n_sites


# nz x ny x nx: columns of planes too thin for the tiles, by themselves and among
# others, and the ones just above; rows of a multiple of 16 whatever the plane
@pytest.mark.parametrize("shapes,used", [
    ([(9000, 5, 7)], 1), ([(5000, 8, 8), (4500, 8, 9)], 1), ([(3000, 12, 12)], 1), ([(400, 150, 5)], 3),
    ([(3000, 150, 5)], 1), ([(600, 300, 6)], 2), ([(5000, 8, 8), (70, 66, 68)], 1),
    ([(300, 8, 8), (70, 66, 68)], 2), ([(4000, 4, 32)], 2), ([(2500, 16, 16)], 2),
])
def test_thin_columns_take_the_one_step_sweep_with_the_same_bits(lb, shapes, used):
    geoms = [_geom(sh, sum(sh)) for sh in shapes]
    gs = [(0.2, 0.1, -0.3)] * len(geoms)
    out = []
    for multi in (0, 2):
        with _solver(lb, 0, geoms, (0, 0, 0), gs[0], _wave("pgse", 10)) as s:
            s.set_option(lb.OPT_MULTI_STEP, multi)
            fields = [torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda") for g in geoms]
            s.run_batch(lb.Solver.members(gs, list(range(len(geoms))), 0.03), fields=fields)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (used if multi == 0 else 2)
            out.append([v.cpu().numpy() for v in fields])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_batch_members_end_on_either_step_and_runs_continue_in_any_split(lb):
    geoms = [_geom((24, 20, 33), 5), _geom((9, 41, 16), 6), _geom((48, 16, 16), 7)]
    n = 21
    f = _wave("pgse", n)
    waves = [None, _wave("pgse", 10), _wave("cos", 11), _wave("pgse", 1), None, _wave("pgse", 20)]
    gs = [(0.2, 0.1, 0.0), (0.0, 0.3, 0.1), (0.1, 0.1, 0.1), (0.3, 0.0, 0.0), (0.0, 0.0, 0.4), (0.2, 0.0, 0.2)]
    geo = [0, 1, 2, 0, 2, 1]
    res = []
    for kernel in (0, 1):
        with _solver(lb, kernel, geoms, (0, 0, 0), gs[0], f) as s:
            fields = [torch.zeros(geoms[i].n_sites, dtype=torch.complex64, device="cuda") for i in geo]
            m = lb.Solver.members(gs, geo, [0.03, 0.0, INF, 0.1, 0.03, 0.2])
            r = s.run_batch(m, waveforms=waves, fields=fields)
            q = s.run_batch(m, waveforms=waves, fields=fields, series=True)
            torch.cuda.synchronize()
            sums = [float(v.abs().sum()) for v in fields]
            res.append(([v.cpu().numpy() for v in fields], r["Z"], q["Z"], sums))
    for a, b in zip(res[0][0], res[1][0]):
        assert np.array_equal(a, b)
    assert np.all(np.abs(res[0][1] - res[1][1]) <= 2.0 ** -22 * np.array(res[0][3]))
    assert np.array_equal(res[0][1], res[0][2])
    # the same run stepped by hand
    g = geoms[0]
    ref = None
    for split in ([21], [1, 1, 19], [2, 17, 2], [3, 16, 1, 1], [20, 1]):
        with _solver(lb, 0, [g], (0, 0, 0), gs[0], f) as s:
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            s.set_field(fld)
            s.prepare()
            for k in split:
                s.advance(k)
            torch.cuda.synchronize()
            v = fld.cpu().numpy()
        ref = v if ref is None else ref
        assert np.abs(ref).max() > 0 and np.array_equal(ref, v)


# one context, one grid after the other: growing and shrinking, other tiles, batches,
# on-chip grids in between (the tensor maps are rewritten where they lie)
TURNS = [[(37, 23, 31)], [(70, 66, 68)], [(90, 75, 117)], [(4, 300, 300), (70, 66, 68), (66, 70, 81)], [(24, 24, 24)],
         [(75, 90, 117)], [(70, 66, 68), (66, 70, 81)], [(64, 48, 160)], [(70, 66, 68)]]


@pytest.mark.parametrize("multi", [0, 2])
def test_one_context_over_many_grids_gives_what_a_fresh_one_gives(lb, multi):
    gG = (0.2, 0.1, -0.3)

    def job(s, shapes):
        geoms = [_geom(sh, sum(sh)) for sh in shapes]
        for i, g in enumerate(geoms):
            (s.add_geometry if i else s.set_geometry)(g.labels, g.phase_of_label, g.dx, (0, 0, 0))
        fields = [torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda") for g in geoms]
        r = s.run_batch(lb.Solver.members([gG] * len(geoms), list(range(len(geoms))), 0.03), fields=fields)
        torch.cuda.synchronize()
        return [v.cpu().numpy() for v in fields], np.asarray(r["Z"])

    with _solver(lb, 0, [_geom((8, 8, 8), 1)], (0, 0, 0), gG, _wave("pgse", 9)) as s:
        s.set_option(lb.OPT_MULTI_STEP, multi)
        for shapes in TURNS:
            got = job(s, shapes)
            with _solver(lb, 0, [_geom((8, 8, 8), 1)], (0, 0, 0), gG, _wave("pgse", 9)) as fresh:
                fresh.set_option(lb.OPT_MULTI_STEP, multi)
                want = job(fresh, shapes)
            for a, b in zip(got[0], want[0]):
                assert np.array_equal(a, b), shapes
            assert np.array_equal(got[1], want[1]), shapes


# steps by themselves take the one-step sweep: the state changes its layout there and back
@pytest.mark.parametrize("shape,bc,gG", [((37, 23, 31), (0, 0, 0), (0.2, 0.1, -0.3)), ((20, 34, 32), (1, 0, 0), (0.4, 0.0, 0.0)),
                                         ((8, 4, 4), (0, 1, 1), (0.3, 0.0, 0.0)), ((33, 40, 35), (1, 1, 0), (0.0, 0.0, 0.3))])
def test_runs_advanced_step_by_step_give_the_same_bits(lb, shape, bc, gG):
    geoms, n = [_geom(shape, 3), _geom((9, 10, 11), 4)], 30
    m = lb.Solver.members([gG, gG, (0.0, 0.0, 0.0)], [0, 1, 0], [0.03, INF, 0.1])
    ref = None
    for kernel, split in ((1, [30]), (0, [30]), (0, [1] * 30), (0, [10] + [1] * 7 + [8, 1, 1, 1, 2]),
                          (0, [1, 1, 2, 2, 2, 1, 3, 1, 1, 1, 15]), (0, [2, 1, 9, 1, 1, 16]), (0, [1, 29]), (0, [29, 1])):
        assert sum(split) == n
        with _solver(lb, kernel, geoms, bc, gG, _wave("cos", n)) as s:
            s.prepare(m)
            z = [s.advance(k, True, 3) for k in split][-1][:, :2]
            with _solver(lb, kernel, geoms[:1], bc, gG, _wave("cos", n)) as one:
                fld = torch.zeros(geoms[0].n_sites, dtype=torch.complex64, device="cuda")
                one.set_field(fld)
                one.prepare()
                zs = [one.advance(k, True) for k in split][-1][0, :2]
                torch.cuda.synchronize()
                v = fld.cpu().numpy()
        if ref is None:
            ref = (z, v)
        assert np.array_equal(ref[1], v) and np.abs(v).max() > 0, split
        tol = 2.0 ** -22 * geoms[0].n_sites
        assert np.abs(z - ref[0]).max() <= tol, split
        assert np.abs(zs - ref[0][0]).max() <= tol, split


# few steps do not pay for the plan: four for the resident sweep and one more for each
# 52000 sites, ten or 16 M site-steps for the two-step sweep; a caller's choice is taken
@pytest.mark.parametrize("shape,n,multi,used", [
    ((12, 13, 14), 3, 0, 1), ((12, 13, 14), 4, 0, 3), ((12, 13, 14), 2, 3, 3), ((40, 41, 42), 4, 0, 1), ((40, 41, 42), 5, 0, 3),
    ((70, 66, 68), 9, 0, 1), ((70, 66, 68), 10, 0, 2),
    ((70, 66, 68), 2, 2, 2), ((200, 200, 200), 2, 0, 2), ((199, 200, 200), 2, 0, 1), ((12, 13, 14), 1, 0, 1),
])
def test_runs_of_few_steps(lb, shape, n, multi, used):
    g = _geom(shape, 8)
    out = []
    for opt in (multi, 1):
        with _solver(lb, 0, [g], (0, 0, 0), (0.2, 0.1, 0.3), _wave("cos", n)) as s:
            s.set_option(lb.OPT_MULTI_STEP, opt)
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            s.run(field=fld)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (used if opt == multi else 1)
            out.append(fld.cpu().numpy())
    assert np.array_equal(out[0], out[1])


# the tuner times one-step sweeps: whole runs of the others do not wait for it
@pytest.mark.parametrize("shape,multi,tuned", [((70, 66, 68), 0, False), ((20, 24, 32), 0, False), ((70, 66, 68), 1, True)])
def test_the_tuner_is_left_out_of_runs_that_take_none_of_its_sweeps(lb, shape, multi, tuned):
    g = _geom(shape, 8)
    out = []
    for tune in (0, 1):
        with _solver(lb, 0, [g], (0, 0, 0), (0.2, 0.1, 0.3), _wave("pgse", 20)) as s:
            s.set_option(lb.OPT_MULTI_STEP, multi)
            s.set_option(lb.OPT_AUTOTUNE, tune)
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            s.run(field=fld)
            torch.cuda.synchronize()
            out.append((fld.cpu().numpy(), s.launch_count()))
    assert np.array_equal(out[0][0], out[1][0])
    assert (out[1][1] > out[0][1] + 50) if tuned else out[1][1] == out[0][1]

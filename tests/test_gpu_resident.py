"""The resident sweep (all steps of a run in one launch) against the one-step
sweeps: the same bits in the field; the signal is summed from the same FP32
thread sums, so it differs by FP64 rounding only (1e-13 of the sum of |M|);
the series is summed in FP64 throughout, so it differs by the FP32 rounding of
the one-step sweep's thread sums (three sites at most: 2^-22 of the sum)."""
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


def _geom(shape, seed):
    rng = np.random.default_rng(seed)
    coarse = rng.integers(0, 3, size=[(n + 2) // 3 for n in shape])
    lab = np.kron(coarse, np.ones((3, 3, 3), int))[:shape[0], :shape[1], :shape[2]]
    return synth.Geometry(np.ascontiguousarray(lab, np.int32), np.arange(3, dtype=np.uint8), 0.5)


def _solver(lb, multi, geoms, bc, gG, f, kap, lattice):
    s = lb.Solver(0)
    s.set_option(lb.OPT_MULTI_STEP, multi)
    s.set_option(lb.OPT_LATTICE, lattice)
    for i, g in enumerate(geoms):
        (s.add_geometry if i else s.set_geometry)(g.labels, g.phase_of_label, g.dx, bc)
    s.set_phases([2.0, 1.0, 1.5], [80.0, 50.0, INF])
    s.set_permeability(kap)
    s.set_sequence(0.01, f, gG)
    return s


def _wave(kind, n):
    f = np.zeros(n)
    f[:max(1, n // 3)] = 1.0
    f[n - max(1, n // 3):] = -1.0
    return f if kind == "pgse" else np.cos(np.arange(n) * 0.7)


# one block, one row or plane a block, ragged cuts, faces of every kind, the
# largest blocks (2048 sites), both lattices
CASES = [
    ((1, 1, 1), (0, 0, 0), (0.3, 0.2, 0.1), "pgse", 7, 0),
    ((2, 1, 9), (0, 0, 0), (0.3, 0.0, 0.1), "cos", 5, 0),
    ((7, 5, 3), (1, 1, 1), (0.0, 0.2, 0.0), "pgse", 6, 0),
    ((32, 32, 32), (0, 0, 0), (0.2, 0.1, -0.3), "pgse", 40, 0),
    ((31, 29, 33), (1, 0, 0), (0.4, 0.0, 0.0), "cos", 17, 0),
    ((23, 41, 16), (0, 1, 1), (0.3, 0.0, 0.0), "pgse", 20, 0),
    ((57, 57, 57), (0, 0, 0), (0.1, -0.2, 0.1), "pgse", 12, 0),
    ((64, 64, 64), (1, 1, 1), (0.0, 0.0, 0.3), "pgse", 9, 0),
    ((1, 200, 200), (0, 0, 0), (0.3, 0.2, 0.0), "pgse", 30, 1),
    ((1, 61, 500), (1, 1, 0), (0.0, 0.2, 0.0), "cos", 11, 1),
    ((1, 3, 1024), (0, 1, 0), (0.1, 0.0, 0.0), "pgse", 4, 1),
    # strips: one to eight rows, two and three columns a thread, ragged
    ((1, 140, 1150), (0, 0, 0), (0.3, 0.1, 0.0), "pgse", 7, 1),
    ((1, 152, 2100), (1, 0, 0), (0.2, 0.0, 0.0), "pgse", 5, 1),
    ((1, 1000, 1000), (1, 1, 0), (0.2, 0.0, 0.0), "pgse", 24, 1),
    ((1, 1216, 700), (0, 0, 0), (0.1, 0.3, 0.0), "cos", 9, 1),
    ((1, 600, 1500), (0, 1, 0), (0.0, 0.3, 0.0), "pgse", 8, 1),
]


@pytest.mark.parametrize("shape,bc,gG,wave,n,lattice", CASES)
@pytest.mark.parametrize("kap", [0.03, 0.0, INF])
def test_resident_sweep_gives_the_one_step_bits(lb, shape, bc, gG, wave, n, lattice, kap):
    g = _geom(shape, sum(shape))
    f = _wave(wave, n)
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, [g], bc, gG, f, kap, lattice) as s:
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            r = s.run(field=fld, series=True)
            q = s.run(field=fld)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi or shape[2] > 1536 and min(shape) == 1 else 3)
            out.append((fld.cpu().numpy(), r, q))
    assert np.array_equal(out[0][0], out[1][0])
    total = np.abs(out[0][0]).sum()
    assert abs(out[0][2]["Z"] - out[1][2]["Z"]) <= 1e-13 * total
    assert np.abs(out[0][1]["series"] - out[1][1]["series"]).max() <= 2.0 ** -22 * g.n_sites


def test_resident_batch_with_own_echoes_and_any_split(lb):
    geoms = [_geom((24, 20, 33), 5), _geom((9, 41, 16), 6), _geom((12, 16, 16), 7)]
    n = 21
    f = _wave("pgse", n)
    waves = [None, _wave("pgse", 10), _wave("cos", 11), _wave("pgse", 1), None]
    gs = [(0.2, 0.1, 0.0), (0.0, 0.3, 0.1), (0.1, 0.1, 0.1), (0.3, 0.0, 0.0), (0.0, 0.0, 0.4)]
    geo = [0, 1, 2, 0, 2]
    res = []
    for multi in (0, 1):
        with _solver(lb, multi, geoms, (0, 0, 0), gs[0], f, 0.03, 0) as s:
            fields = [torch.zeros(geoms[i].n_sites, dtype=torch.complex64, device="cuda") for i in geo]
            r = s.run_batch(lb.Solver.members(gs, geo, [0.03, 0.0, INF, 0.1, 0.03]), waveforms=waves, fields=fields)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi else 3)
            res.append(([v.cpu().numpy() for v in fields], r["Z"], np.array([float(v.abs().sum()) for v in fields])))
    for a, b in zip(res[0][0], res[1][0]):
        assert np.array_equal(a, b)
    assert np.all(np.abs(res[0][1] - res[1][1]) <= 1e-13 * res[0][2])
    g = geoms[0]
    ref = None
    for split in ([21], [1, 1, 19], [2, 17, 2], [20, 1]):   # one step by itself: the one-step sweep
        with _solver(lb, 0, [g], (0, 0, 0), gs[0], f, 0.03, 0) as s:
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            s.set_field(fld)
            s.prepare()
            for k in split:
                s.advance(k)
            torch.cuda.synchronize()
            v = fld.cpu().numpy()
        ref = v if ref is None else ref
        assert np.abs(ref).max() > 0 and np.array_equal(ref, v)


# blocks of two and more layers, the rule's second neighbours across every kind
# of face; random positions (any link, any compartment)
@pytest.mark.parametrize("shape,bc,gG,wave,n,lattice", [
    ((12, 10, 9), (0, 0, 0), (0.3, 0.2, 0.1), "pgse", 9, 0),
    ((24, 31, 20), (1, 0, 1), (0.3, 0.0, 0.0), "cos", 8, 0),
    ((2, 3, 5), (0, 0, 0), (0.2, 0.1, 0.3), "pgse", 6, 0),
    ((1, 200, 200), (0, 0, 0), (0.3, 0.2, 0.0), "pgse", 30, 1),
    ((1, 65, 130), (1, 1, 0), (0.0, 0.2, 0.0), "cos", 21, 1),
    ((1, 37, 22), (0, 1, 0), (0.1, 0.0, 0.0), "pgse", 14, 1),
])
def test_resident_sweep_with_membrane_positions(lb, shape, bc, gG, wave, n, lattice):
    """Against the register sweep's position rule: the same bits."""
    g = _geom(shape, sum(shape) + 1)
    f = _wave(wave, n)
    delta = np.random.default_rng(3).uniform(0.1, 0.9, size=(6, *shape)).astype(np.float32)
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, [g], bc, gG, f, 0.05, lattice) as s:
            s.set_link_distances(delta)
            fld = torch.zeros(g.n_sites, dtype=torch.complex64, device="cuda")
            r = s.run(field=fld, series=True)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi else 3)
            assert s.get_option(lb.OPT_KERNEL_USED) == 1
            out.append((fld.cpu().numpy(), r))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][1]["series"] - out[1][1]["series"]).max() <= 2.0 ** -22 * g.n_sites


# one and two sites a thread, one segment and several, a short last one, faces of
# every kind, two members of different geometry
@pytest.mark.parametrize("shapes,bc,gG,wave,n,every", [
    ([(48, 48, 48)], (0, 0, 0), (0.3, 0.2, 0.1), "pgse", 30, 8),
    ([(20, 24, 32)], (0, 0, 0), (0.2, -0.3, 0.1), "cos", 17, 64),
    ([(9, 31, 48)], (1, 1, 1), (0.0, 0.0, 0.4), "pgse", 21, 5),
    ([(40, 30, 16)], (1, 0, 1), (0.4, 0.0, 0.0), "pgse", 12, 4),
    ([(16, 32, 16), (7, 9, 48)], (0, 0, 0), (0.1, 0.2, 0.1), "pgse", 19, 6),
])
def test_resident_gradient_is_the_bulk_copy_one(lb, shapes, bc, gG, wave, n, every):
    """Signal, gradients: the same arithmetic and the same groups of partial
    sums, so the same numbers (1e-12 for the FP64 sums of the signal)."""
    geoms = [_geom(s, sum(s)) for s in shapes]
    f = _wave(wave, n)
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, geoms, bc, gG, f, 0.05, 0) as s:
            m = lb.Solver.members([gG] * len(geoms), list(range(len(geoms))), 0.05)
            c0 = s.launch_count()
            r = s.grad_batch(m, checkpoint_every=every)
            out.append((r, s.launch_count() - c0))
    assert out[0][1] < out[1][1]   # it ran
    assert np.allclose(out[0][0]["Z"], out[1][0]["Z"], rtol=1e-12, atol=0)
    for k in ("dD", "dT2", "dkappa"):
        a, b = out[0][0][k], out[1][0][k]
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), (k, a, b)


# segments longer than a launch of the resident adjoint (256 steps): the same numbers,
# and no more memory than the levels and the sensitivities of 256 steps
@pytest.mark.parametrize("n,every", [(600, 600), (513, 300), (256, 256)])
def test_resident_gradient_of_long_segments(lb, n, every):
    g = _geom((31, 32, 48), 4)
    f = 0.02 * _wave("cos", n)
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, [g], (0, 0, 0), (0.3, 0.2, 0.1), f, 0.05, 0) as s:
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            out.append(s.grad(checkpoint_every=every))
            held = before - torch.cuda.mem_get_info()[0]
            n_ck = -(-n // every)
            levels = 2 + n_ck + n_ck * every + 1   # state, checkpoints, segments (all kept at most)
            assert held <= g.n_sites * (56 * levels + 12 * 256 + 8) + (64 << 20)
    assert np.allclose(out[0]["Z"], out[1]["Z"], rtol=1e-12, atol=0)
    for k in ("dD", "dT2", "dkappa"):
        a, b = np.asarray(out[0][k]), np.asarray(out[1][k])
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), (k, a, b)


# as many members as SMs, of one shape and of mixed ones in any order; one too many blocks
@pytest.mark.parametrize("shapes,used", [
    ([(12, 12, 12)] * 150, 3), ([(6, 7, 8), (6, 7, 8), (9, 5, 7), (6, 7, 8)] * 30, 3), ([(14, 14, 14)] * 100, 2),
    ([(20, 20, 20), (8, 9, 10), (20, 20, 20)] * 8, 3), ([(8, 9, 10)] * 153, 1),
])
def test_resident_batches_of_many_members(lb, shapes, used):
    geoms = [_geom(sh, sum(sh)) for sh in sorted(set(shapes))]
    which = [sorted(set(shapes)).index(sh) for sh in shapes]
    rng = np.random.default_rng(2)
    gs = [tuple(v) for v in rng.normal(size=(len(shapes), 3)) * 0.2]
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, geoms, (0, 0, 0), gs[0], _wave("pgse", 12), 0.03, 0) as s:
            fields = [torch.zeros(geoms[i].n_sites, dtype=torch.complex64, device="cuda") for i in which]
            s.run_batch(lb.Solver.members(gs, which, 0.03), fields=fields)
            torch.cuda.synchronize()
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi else used)
            out.append([v.cpu().numpy() for v in fields])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


# every step's signal is made of the one-step sweep's thread sums; free diffusion along x,
# where the roundings of all rows are alike and add up; several launches (32 steps at
# least of what 256 MB hold), blocks and strips, members of two sizes
@pytest.mark.parametrize("shapes,lattice,n", [([(23, 41, 46)], 0, 60), ([(32, 32, 32)], 0, 60), ([(1, 500, 1000)], 1, 75),
                                              ([(20, 24, 33), (7, 9, 10)], 0, 20), ([(1, 61, 90)], 1, 40)])
def test_resident_series_is_the_one_step_series(lb, shapes, lattice, n):
    geoms = [synth.Geometry(np.zeros(sh, np.int32), np.zeros(1, np.uint8), 1.0) for sh in shapes]
    out = []
    for multi in (0, 1):
        with _solver(lb, multi, geoms, (0, 0, 0), (0.4, 0.0, 0.0), _wave("pgse", n), INF, lattice) as s:
            m = lb.Solver.members([(0.4, 0.0, 0.0), (0.1, 0.0, 0.0)] * len(geoms), list(range(len(geoms))) * 2, INF)
            r = s.run_batch(m, series=True)
            assert s.get_option(lb.OPT_MULTI_STEP_USED) == (1 if multi else 3)
            out.append(np.asarray(r["series"]))
    assert np.abs(out[1]).min() > 0
    strips = lattice == 1 and geoms[0].n_sites > 400000
    assert np.abs(out[0] - out[1]).max() <= (2.0 ** -22 if strips else 1e-13) * max(g.n_sites for g in geoms)

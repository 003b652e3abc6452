"""The resident FP64 cells, the long candidate lists of the resident FP32 cells
and the truth DEM's lists against the oracle, at the sizes where their
branches part.  Tolerances as in the parity tests: 1e-10 (FP64) and 1e-4
(FP32), relative, per moment column."""
import numpy as np
import pytest

from paper_2303_07819_gb300 import inputs as I
from tests.parity import rel_errors, report

pytestmark = pytest.mark.gpu

TOL = {0: (1e-4, 1e-6), 1: (1e-10, 1e-12)}     # precision: tolerance, floor


@pytest.fixture(scope="module")
def ms():
    from paper_2303_07819_gb300 import msdem
    msdem.load()
    return msdem


def soft(nx, L):
    """The square's constants with a soft, undamped contact law: floes may
    overlap by tens of percent without flying apart."""
    p = dict(I.square_4x4()["params"], nx=nx, ny=nx, Lx=L, Ly=L, E=20.0, G=10.0, eta=0.0, N0=10, n_t=5)
    p["modes"] = I.psi_sin_sin_modes(0.1, L)
    return p


def crowd(seed, n, side, cover):
    rng = np.random.default_rng(seed)
    r0 = np.sqrt(cover * side * side / (np.pi * max(n, 1)))
    return I.random_cell_floes(rng, n, side, 0.5 * min(r0, 0.16 * side), min(r0, 0.16 * side))


def join(parts):
    return {k: np.concatenate([f[k] for f in parts]) for k in I.random_cell_floes(np.random.default_rng(0), 1, 1.0, 0.1, 0.2)}


def ring(n, side, big, small):
    """One floe of radius `big` with n small ones touching it all round, in as many rings as they need."""
    f = I.random_cell_floes(np.random.default_rng(n), n + 1, side, 0.9 * small, small)
    f["r"][0] = big
    f["x"][0] = f["y"][0] = 0.5 * side
    per = max(3, int(2 * np.pi * (big + small) / (2.02 * small)))
    k = np.arange(n)
    rad = big + (0.9 + 1.5 * (k // per)) * small
    ang = 2 * np.pi * (k % per + 0.5 * (k // per % 2)) / per
    f["x"][1:] = 0.5 * side + rad * np.cos(ang)
    f["y"][1:] = 0.5 * side + rad * np.sin(ang)
    return f


@pytest.mark.parametrize("n", [1, 2, 16, 17, 31, 33, 65, 129, 300, 1024, 1025])
@pytest.mark.parametrize("threads,persistent", [(64, 0), (128, 1), (256, 0)])
def test_fp64_cells(orc, ms, n, threads, persistent):
    """Cells of n floes (1025: the all-pairs kernel), beside cells of 3, none
    and 1, across two coarse steps, in one call and in steps of 1 and 7."""
    if n > 300 and threads != 128:
        pytest.skip("one block size for the large cells")
    side = 25e3
    parts = [crowd(n, n, side, 0.7), crowd(7, 3, side, 0.3), crowd(8, 1, side, 0.1)]
    parts[1]["x"] += side
    parts[2]["x"] += side
    parts[2]["y"] += side
    f, p = join(parts), soft(2, 2 * side)
    o = orc.Model(p, f)
    a, b = ms.Model(p, f, ms.MS_FP64), ms.Model(p, f, ms.MS_FP64)
    for m in (a, b):
        m.set_launch(0, threads, persistent, 1.0)
    o.step(10.0, 23)
    a.step(10.0, 23)
    for k in (1, 7, 1, 14):
        b.step(10.0, k)
    e = rel_errors(a.moments(), o.moments(), p, TOL[1][1])
    assert e.max() <= TOL[1][0], report(e)
    fa, fb = a.floes(), b.floes()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)
    assert np.array_equal(a.coupling()["window"], b.coupling()["window"])


@pytest.mark.parametrize("n,big,small", [(11, 3000.0, 400.0), (13, 3000.0, 400.0), (24, 4000.0, 400.0), (26, 4000.0, 400.0),
                                         (200, 5000.0, 150.0), (300, 5000.0, 150.0), (600, 5000.0, 100.0)])
def test_fp32_long_lists(orc, ms, n, big, small):
    """A large floe with n partners: lists up to the slots of a build's first
    sort, beyond them, and long enough for a whole warp to walk."""
    side = 25e3
    f, p = ring(n, side, big, small), soft(1, side)
    o, g = orc.Model(p, f), ms.Model(p, f, ms.MS_FP32)
    o.step(10.0, 23)
    g.step(10.0, 23)
    e = rel_errors(g.moments(), o.moments(), p, TOL[0][1])
    assert e.max() <= TOL[0][0], report(e)


@pytest.mark.parametrize("n", [40, 250, 500, 900])
def test_fp32_lists_that_do_not_fit(orc, ms, n):
    """So crowded that a group's lists exceed their room: every pair of the
    cell is tested."""
    side = 25e3
    f, p = crowd(n, n, side, 5.0), soft(1, side)
    o, g = orc.Model(p, f), ms.Model(p, f, ms.MS_FP32)
    o.step(10.0, 12)
    g.step(10.0, 12)
    e = rel_errors(g.moments(), o.moments(), p, TOL[0][1])
    assert e.max() <= TOL[0][0], report(e)


@pytest.mark.parametrize("nx,n", [(1, 400), (3, 30), (6, 3)])
def test_fp32_uncoupled_split(ms, nx, n):
    """Uncoupled steps short of a whole interval give the same floes however
    they are split into calls, to the last bit."""
    side = 25e3
    parts = [crowd(c, n, side, 0.7) for c in range(nx * nx)]
    for c, f in enumerate(parts):
        f["x"] += side * (c % nx)
        f["y"] += side * (c // nx)
    f, p = join(parts), dict(soft(nx, nx * side), couple=0)
    a, b = ms.Model(p, f, ms.MS_FP32), ms.Model(p, f, ms.MS_FP32)
    a.step(10.0, 61)
    for k in (1, 1, 7, 33, 19):
        b.step(10.0, k)
    fa, fb = a.floes(), b.floes()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)
    assert np.array_equal(a.moments(), b.moments())


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,big,small", [(1, 3000.0, 400.0), (15, 3000.0, 400.0), (17, 3000.0, 400.0), (60, 5000.0, 300.0),
                                         (70, 5000.0, 300.0), (150, 6000.0, 150.0)])
def test_truth_lists(orc, ms, precision, n, big, small):
    """Truth lists of up to 16, up to 64 and more candidates; runs split
    anywhere give the same floes."""
    L = 100e3
    f, p = ring(n, L, big, small), dict(soft(4, L), couple=0)
    o = orc.Truth(p, f)
    a, b = ms.Model(p, f, precision), ms.Model(p, f, precision)
    o.step(10.0, 23)
    a.truth_step(10.0, 23)
    for k in (1, 7, 15):
        b.truth_step(10.0, k)
    e = rel_errors(a.truth_moments(), o.moments(), p, TOL[precision][1])
    assert e.max() <= TOL[precision][0], report(e)
    fa, fb = a.truth_floes(), b.truth_floes()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)

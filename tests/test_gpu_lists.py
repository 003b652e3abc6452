"""Candidate lists of the resident FP64 cells, the resident FP32 cells and the
truth DEM where their upkeep is at its limits: rebuilt at every step, longer
than their room, of floes far from the mean speed, radius or density.
Tolerances as in the parity tests: 1e-10 (FP64) and 1e-4 (FP32), relative,
per moment column."""
import subprocess
import sys
import time

import numpy as np
import pytest

from paper_2303_07819_gb300.inputs import square_4x4
from tests.conftest import ROOT
from tests.parity import rel_errors, report
from tests.test_gpu_runs import TOL, crowd, join, ring, soft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ms():
    from paper_2303_07819_gb300 import msdem
    msdem.load()
    return msdem


def same_floes(fa, fb):
    return all(np.array_equal(fa[k], fb[k]) for k in fa)


@pytest.mark.parametrize("n", [5, 32, 40, 100])
@pytest.mark.parametrize("threads", [64, 256])
def test_fp64_lists_made_at_every_step(orc, ms, n, threads):
    """A gradual update at every step of the second and third interval: each
    step searches anew, and the warp then takes pairs of lists that other
    lanes have just written."""
    side = 25e3
    parts = [crowd(n + c, n, side, 1.5) for c in range(4)]
    for c, q in enumerate(parts):
        q["x"] += side * (c % 2)
        q["y"] += side * (c // 2)
    f, p = join(parts), dict(soft(2, 2 * side), n_t=1)
    o = orc.Model(p, f)
    a, b = ms.Model(p, f, ms.MS_FP64), ms.Model(p, f, ms.MS_FP64)
    for m in (a, b):
        m.set_launch(0, threads, 0, 1.0)
    o.step(10.0, 23)
    a.step(10.0, 23)
    for k in (1, 2, 20):
        b.step(10.0, k)
    e = rel_errors(a.moments(), o.moments(), p, TOL[1][1])
    assert e.max() <= TOL[1][0], report(e)
    assert same_floes(a.floes(), b.floes())


def packed(n, L, seed=5):
    """n floes of about 0.3 spacings on a jittered lattice over an L x L domain, at rest."""
    rng = np.random.default_rng(seed)
    k = int(np.ceil(np.sqrt(n)))
    d = L / k
    i = np.arange(n)
    f = {key: np.zeros(n) for key in ("x", "y", "theta", "u", "v", "omega", "r", "h")}
    f["x"] = (i % k + 0.5 + rng.uniform(-0.2, 0.2, n)) * d
    f["y"] = (i // k + 0.5 + rng.uniform(-0.2, 0.2, n)) * d
    f["r"] = rng.uniform(0.25, 0.35, n) * d
    f["h"] = rng.uniform(0.5, 2.0, n)
    return f


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [90, 900, 3000])
def test_truth_fast_floes(orc, ms, precision, n):
    """All floes at tens of metres a step and one faster still: wider
    skins than a list may have, so lists are made again every few steps.  The
    oracle's moments, and the same floes however the run is split."""
    L = 30e3
    f, p = packed(n, L), dict(soft(2, L), couple=0)
    rng = np.random.default_rng(n)
    f["u"], f["v"] = rng.uniform(-40.0, 40.0, n), rng.uniform(-40.0, 40.0, n)
    f["u"][n // 2] = 100.0
    o = orc.Truth(p, f)
    a, b = ms.Model(p, f, precision), ms.Model(p, f, precision)
    o.step(0.5, 24)
    a.truth_step(0.5, 24)
    for k in (1, 7, 16):
        b.truth_step(0.5, k)
    e = rel_errors(a.truth_moments(), o.moments(), p, TOL[precision][1])
    assert e.max() <= TOL[precision][0], report(e)
    assert same_floes(a.truth_floes(), b.truth_floes())


@pytest.mark.parametrize("precision", [0, 1])
def test_truth_diverged_state(ms, precision):
    """Every floe at 1e12 m/s: the speeds turn inf and NaN within a few steps,
    from which no list may grow with the number of floes.  60,000 floes, 200
    steps: with lists of a few neighbours, made at every step, some 0.1 ms a
    step; had every floe the others as candidates, 4e9 tests a step.  The
    step reports MS_ERR_UNSTABLE and the context stays usable."""
    n, L = 60_000, 300e3
    f, p = packed(n, L), dict(soft(8, L), couple=0)
    f["u"][:] = 1.0e12
    m = ms.Model(p, f, precision)
    t = time.perf_counter()
    with pytest.raises(ms.MsError) as e:
        m.truth_step(10.0, 200)
    assert e.value.code == -3, str(e.value)
    assert time.perf_counter() - t < 1.0
    f["u"][:] = 0.0
    m = ms.Model(p, f, precision)
    m.truth_step(10.0, 3)
    assert np.all(np.isfinite(m.truth_moments()))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,small", [(63, 300.0), (64, 300.0), (65, 250.0), (130, 200.0), (220, 80.0), (230, 80.0), (900, 20.0)])
def test_truth_long_lists(orc, ms, precision, n, small):
    """Two large floes of one warp, one of them across the domain's corner,
    each with up to n partners: lists of just up to 64, portions of 64 of longer
    ones, and more partners than one search of the warp holds.  The oracle's
    moments, and the same floes however the run is split."""
    L = 100e3
    parts = [ring(n, L, 6000.0, small), ring(n, L, 5900.0, small)]
    parts[0]["x"] = np.mod(parts[0]["x"] + 0.5 * L, L)
    parts[0]["y"] = np.mod(parts[0]["y"] + 0.5 * L, L)
    f = join(parts)
    order = np.r_[0, n + 1, 1:n + 1, n + 2:2 * n + 2]
    f, p = {k: v[order] for k, v in f.items()}, dict(soft(4, L), couple=0)
    o = orc.Truth(p, f)
    a, b = ms.Model(p, f, precision), ms.Model(p, f, precision)
    o.step(10.0, 23)
    a.truth_step(10.0, 23)
    for k in (1, 7, 15):
        b.truth_step(10.0, k)
    e = rel_errors(a.truth_moments(), o.moments(), p, TOL[precision][1])
    assert e.max() <= TOL[precision][0], report(e)
    assert same_floes(a.truth_floes(), b.truth_floes())


@pytest.mark.parametrize("precision", [0, 1])
def test_truth_diverged_between_walls(ms, precision):
    """As test_truth_diverged_state, between walls: within two steps all
    floes stand on a wall, some 140 to a bin's side, each with as many
    partners.  20,000 floes, 200 steps: a few ms a step at most."""
    n, L = 20_000, 170e3
    f, p = packed(n, L), dict(soft(8, L), couple=0, walls=1)
    f["u"][:] = 1.0e12
    m = ms.Model(p, f, precision)
    t = time.perf_counter()
    with pytest.raises(ms.MsError) as e:
        m.truth_step(10.0, 200)
    assert e.value.code == -3, str(e.value)
    assert time.perf_counter() - t < 1.0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,r", [(2, 40.0), (500, 50.0), (1500, 60.0), (333, 777.0)])
def test_truth_sparse(orc, ms, precision, n, r):
    """Touching pairs far from each other, up to a million bins to a few
    floes: the oracle's moments, the same floes however the run is split, and
    no call of one step that goes over all bins on the few blocks of the
    floes (which took 2.6 ms; a call costs some 0.05)."""
    L = 100e3
    f, p = packed(n, L), dict(soft(4, L), couple=0)
    f["r"][:] = r
    f["x"][1::2], f["y"][1::2] = np.mod(f["x"][:n - n % 2:2] + 1.9 * r, L), f["y"][:n - n % 2:2]
    o = orc.Truth(p, f)
    a, b = ms.Model(p, f, precision), ms.Model(p, f, precision)
    o.step(10.0, 23)
    a.truth_step(10.0, 23)
    t = []
    for _ in range(23):
        t0 = time.perf_counter()
        b.truth_step(10.0, 1)
        t.append(time.perf_counter() - t0)
    e = rel_errors(a.truth_moments(), o.moments(), p, TOL[precision][1])
    assert e.max() <= TOL[precision][0], report(e)
    assert same_floes(a.truth_floes(), b.truth_floes())
    assert np.median(t) < 1.0e-3


def test_first_calls_of_several_threads(tmp_path):
    """Models of several threads that make a process's first steps together
    (launch sizes and kernel limits are worked out by whoever comes first)
    give the floes of one model stepped alone."""
    prog = tmp_path / "first.py"
    prog.write_text(f"""
import sys, threading
sys.path.insert(0, {ROOT!r})
import numpy as np
from paper_2303_07819_gb300 import msdem as ms
from tests.test_gpu_lists import packed
from tests.test_gpu_runs import soft
ms.load()
out, start = [None] * 8, threading.Barrier(8)
def one(i):
    start.wait()
    m = ms.Model(dict(soft(4, 100e3)), packed(900, 100e3), i % 2)
    start.wait()
    m.truth_step(10.0, 5)
    m.step(10.0, 15)
    out[i] = (m.truth_floes(), m.floes())
th = [threading.Thread(target=one, args=(i,)) for i in range(8)]
[t.start() for t in th]
[t.join() for t in th]
for p in (0, 1):
    m = ms.Model(dict(soft(4, 100e3)), packed(900, 100e3), p)
    m.truth_step(10.0, 5)
    m.step(10.0, 15)
    ref = (m.truth_floes(), m.floes())
    for i in range(p, 8, 2):
        for a, b in zip(out[i], ref):
            assert all(np.array_equal(a[k], b[k]) for k in b), i
print("same")
""")
    r = subprocess.run([sys.executable, str(prog)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout + r.stderr


def test_fp64_autotune_times_what_a_step_makes(ms):
    """The time ms_autotune returns and chooses by is that of the run of an
    interval that ms_step makes, not of a step with a launch, loads, a search
    and moments of its own."""
    s = square_4x4()
    m = ms.Model(s["params"], s["floes"], ms.MS_FP64)
    best = m.autotune(s["dt"], reps=5)
    run = min(m.time_kernel(2, s["dt"], reps=5) for _ in range(5)) / s["params"]["N0"]
    assert 0.7 * run < best < 1.3 * run, (best, run)


@pytest.mark.parametrize("nx,n,sparse", [(1, 250, False), (16, 80, False), (16, 80, True)])
def test_fp32_blocks_of_256_that_test_every_pair(orc, ms, nx, n, sparse):
    """Contacts alone exceed the room of a block's lists (12 candidates a floe
    for 256 floes, 384 hits beyond a floe's first 12), with skins or without:
    a cell of 250 floes with a block of its own, blocks of three crowded
    cells of 80, and of crowded cells beside a sparse one."""
    side = 25e3
    parts, deg = [], []
    for c in range(nx * nx):
        f = crowd(1000 + c, n, side, 0.3 if sparse and c % 3 == 1 else 10.0)
        dx, dy = (f[k][:, None] - f[k][None, :] for k in ("x", "y"))
        dx, dy = dx - side * np.rint(dx / side), dy - side * np.rint(dy / side)
        deg.append((np.hypot(dx, dy) < f["r"][:, None] + f["r"][None, :]).sum(1) - 1)
        f["x"] += side * (c % nx)
        f["y"] += side * (c // nx)
        parts.append(f)
    group = max(1, 256 // n)
    over = []
    for g in range(0, nx * nx - group + 1, group):
        d = np.concatenate(deg[g:g + group])
        over.append(d.sum() > 12 * 256 or np.maximum(d - 12, 0).sum() > 384)
    assert np.mean(over) >= (0.5 if sparse else 1.0)
    f, p = join(parts), dict(soft(nx, nx * side), couple=0)
    o, m = orc.Model(p, f), ms.Model(p, f, ms.MS_FP32)
    o.step(10.0, 12)
    m.step(10.0, 12)
    e = rel_errors(m.moments(), o.moments(), p, TOL[0][1])
    assert e.max() <= TOL[0][0], report(e)


@pytest.mark.parametrize("n", [4096, 4097, 8192, 100_003, 200_000])
def test_moments_of_a_crowded_cell(ms, n):
    """Nearly all floes in one cell, around the 4096 above which a warp merges
    its list, through the allocation-free entry point: the sums of each
    cell's floes, the same twice."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    side, extra = 25e3, 37
    p = dict(soft(2, 2 * side))
    f = {k: rng.uniform(0.5, 1.5, n + extra) for k in ("u", "v", "omega", "r", "h")}
    f["x"] = np.r_[rng.uniform(0, side, n), rng.uniform(side, 2 * side, extra)]
    f["y"] = rng.uniform(0, side, n + extra)
    order = rng.permutation(n + extra)
    dev = {k: torch.tensor(v[order], dtype=torch.float64, device="cuda") for k, v in f.items()}
    fd = torch.tensor(rng.normal(size=(3, n + extra)), dtype=torch.float64, device="cuda")
    out = []
    for _ in range(2):
        o = torch.full((4, 12), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        t = time.perf_counter()
        ms.cell_moments_noalloc(p, n + extra, *(dev[k].data_ptr() for k in ("x", "y", "u", "v", "omega", "r", "h")),
                                fd.data_ptr(), o.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert time.perf_counter() - t < 1.0
        out.append(o.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    m = p["rho_ice"] * np.pi * f["r"] ** 2 * f["h"]
    d = fd.cpu().numpy()[:, np.argsort(order)]
    for c, sel in ((0, slice(0, n)), (1, slice(n, n + extra))):
        ref = [m[sel].sum(), (m * f["u"])[sel].sum(), (m * f["v"])[sel].sum()]
        assert out[0][c, 0] == (n if c == 0 else extra)
        assert np.allclose(out[0][c, 1:4], ref, rtol=1e-11, atol=0)
        assert np.allclose(out[0][c, 9:12], d[:, sel].sum(1), rtol=1e-10, atol=1e-10)
    assert np.all(out[0][2:] == 0)


def test_moments_of_a_diverged_truth_state(ms):
    """The moments of a truth DEM whose FP64 positions are NaN, so that all
    floes count to one cell: an answer in a time of the order of a step's."""
    n, L = 60_000, 300e3
    f, p = packed(n, L), dict(soft(8, L), couple=0)
    f["u"][:] = 1.0e12
    m = ms.Model(p, f, ms.MS_FP64)
    with pytest.raises(ms.MsError):
        m.truth_step(10.0, 100)
    t = time.perf_counter()
    mom = m.truth_moments()
    assert time.perf_counter() - t < 1.0
    assert mom[:, 0].sum() == n

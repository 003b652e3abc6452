"""Candidate lists of the resident FP64 cells, the resident FP32 cells and the
truth DEM where their upkeep is at its limits: rebuilt at every step, longer
than their room, of floes far from the mean speed, radius or density.
Tolerances as in the parity tests: 1e-10 (FP64) and 1e-4 (FP32), relative,
per moment column."""
import numpy as np
import pytest

from tests.parity import rel_errors, report
from tests.test_gpu_runs import TOL, crowd, join, soft

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

"""Time steps far beyond what one Krylov space covers: answered as the oracle does, or reported,
never returned as an unevolved state with status OK.

Ordinary runs: every loop of an exponential is bounded, and a step that is not covered ends in
TTNS_E_NOT_CONVERGED or TTNS_E_NONFINITE.
"""
import numpy as np
import pytest

from oracle.ttns import TTNS
from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


# tensors above and below the Krylov dimension; the cluster's, the sites' and the grid's forms
TREES = {
    "chain": (lambda: W.spin_boson(L=4, d=4, D=4), {}),
    "tiny_chain": (lambda: W.spin_boson(L=2, d=2, D=2), {}),
    "star": (lambda: W.sf_small(seed=7, n_env=3, L=2, d=3, D=3, n_modes=4), {}),
    "star_on_the_grid": (lambda: W.sf_small(seed=7, n_env=3, L=2, d=3, D=3, n_modes=4), dict(grid_threshold=1)),
}


@pytest.mark.parametrize("prec", [ttns.TTNS_FP64, ttns.TTNS_TF32X3])
@pytest.mark.parametrize("name", list(TREES))
def test_a_step_in_the_wrong_unit_is_reported(name, prec):
    make, kw = TREES[name]
    p = make()
    for dt in (1e6, -1e6, 1e300):
        g = ttns.Tree(p, precision=prec, **kw)
        g.step(dt, 1)
        with pytest.raises(ttns.TTNSError) as e:
            g.sync()
        assert e.value.code in (4, 6), str(e.value)
        g.close()


# the oracle's own runs at Krylov tolerances 1e-12 and 1e-14 are 1.3e-10 and 0 apart
@pytest.mark.parametrize("name,dt", [("chain", 20.0), ("tiny_chain", 100.0)])
def test_a_long_step_is_covered_by_substeps(name, dt):
    p = TREES[name][0]()
    o = TTNS(p)
    o.step(dt)
    g = ttns.Tree(p, precision=ttns.TTNS_FP64)
    g.step(dt, 1)
    assert np.abs(g.rho() - o.rho_el()).max() < 1e-7
    g.close()


# narrow and wide spectra for the Krylov dimension, halved times, tolerances near and far from FP32's
# resolution: the spaces end where the oracle's FP64 estimate ends them (its check starts at the
# first step; the library's at a leading-order bound, never later in these runs)
@pytest.mark.parametrize("name,dt,mmax,tol", [("chain", 0.5, 30, 1e-12), ("chain", 20.0, 30, 1e-12), ("chain", 20.0, 6, 1e-9),
                                              ("star", 5.0, 12, 1e-12), ("star", 1.0, 30, 1e-6), ("chain", 0.5, 30, 1e-14)])
def test_krylov_spaces_end_where_the_oracle_ends_them(name, dt, mmax, tol):
    p = TREES[name][0]()
    o = TTNS(p, tol=tol, mmax=mmax)
    o.step(dt)
    g = ttns.Tree(p, precision=ttns.TTNS_FP64, krylov_mmax=mmax, krylov_tol=tol)
    g.step(dt, 1)
    if o.stats.get("not_converged"):  # 64 spaces do not cover the step: the library reports it
        with pytest.raises(ttns.TTNSError) as e:
            g.sync()
        assert e.value.code == 4
        g.close()
        return
    g.sync()
    n = g.counters()["krylov_iters"]
    g.close()
    assert abs(n - o.stats["krylov_iters"]) <= 0.02 * o.stats["krylov_iters"], (n, o.stats)

"""Launches of the persistent kernel: a launch's first operation meets CTAs that have all started,
so that many launches of one step equal one launch of many steps bit for bit.
"""
import numpy as np
import pytest

from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("prec", [ttns.TTNS_FP64, ttns.TTNS_TF32X3])
@pytest.mark.parametrize("kw", [dict(cluster_ctas=16), dict(cluster_ctas=3), dict(cluster_ctas=1),
                                dict(grid_threshold=1)], ids=lambda kw: "-".join(f"{k}{v}" for k, v in kw.items()))
def test_many_short_launches_equal_one_long_launch(kw, prec):
    p = W.sf_small(seed=21, n_env=2, L=3, d=4, D=5, n_modes=6)
    g = ttns.Tree(p, precision=prec, **kw)
    g.step(p.dt, 24)
    ref = g.rho(), g.occupations()
    g.close()
    h = ttns.Tree(p, precision=prec, **kw)
    for _ in range(24):
        h.step(p.dt, 1)
    assert np.array_equal(h.rho(), ref[0]) and np.array_equal(h.occupations(), ref[1])
    h.close()

"""Sets of small trees on every team size with two CTAs per SM and with one, against the FP64 CPU
oracle: peers' shared memory, the draw of the next tree and the site plans of the smaller shared
memory, with neighbouring teams on an SM.

Sizes: one round of trees with two CTAs per SM and two rounds with one, so that the pair is chosen.
Tolerances as in test_gpu_parity.py: 1e-7 in FP64, 1e-6 in the mixed modes.
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


@pytest.mark.parametrize("prec,tol", [(ttns.TTNS_FP64, 1e-7), (ttns.TTNS_TF32X3, 1e-6)])
@pytest.mark.parametrize("ctas,n", [(1, 288), (2, 144), (4, 64), (8, 32), (16, 14)])
def test_pairs_of_teams_on_an_sm_equal_the_oracle(ctas, n, prec, tol):
    ps = [W.sf_small(seed=500 + k, n_env=2, L=2, d=3 + k % 2, D=3 + k % 4, n_modes=4) for k in range(n)]
    pick = [0, n // 2, n - 1]
    pops = {}
    for per_sm, grid in ((2, 0), (1, 152)):
        g = ttns.Tree(ps, precision=prec, cluster_ctas=ctas, grid_ctas=grid)
        assert g.ctas_per_sm() == per_sm
        for _ in range(2):
            g.step(ps[0].dt, 1)
        pops[per_sm] = np.array([g.populations(k) for k in range(n)])
        occ = {k: g.occupations(k) for k in pick}
        g.close()
        for k in pick:
            o = TTNS(ps[k])
            for _ in range(2):
                o.step(ps[k].dt)
            assert np.abs(pops[per_sm][k] - o.populations()).max() < tol, k
            np.testing.assert_allclose(occ[k], o.occupations(), atol=10 * tol)
    assert np.abs(pops[1] - pops[2]).max() < tol

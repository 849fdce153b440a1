"""Rounding of the mixed modes' FP32 products: one step of stars of 4 x 3 sites, against the FP64
path of the same tree (1e-14 from the exact step), as the geometric mean of the relative error of
rho_S over 48 Hamiltonians.

The products sum 16 terms at a time.  With four accumulators per output the mean is 1.6e-8, with one
chain of additions 2.1e-8; runs with other roundings of the same kind scatter by 7 % around
these.  1.9e-8 lies between them.
"""
import numpy as np
import pytest

from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def test_products_of_a_star_keep_several_accumulators():
    err = []
    for seed in range(100, 148):
        p = W.singlet_fission(seed=seed, n_env=4, L=3, d=8, D=16, n_modes=6, dt=0.5, n_steps=1)
        rho = []
        for prec in (ttns.TTNS_FP64, ttns.TTNS_TF32X3):
            g = ttns.Tree(p, precision=prec)
            g.step(p.dt, 1)
            rho.append(g.rho())
            g.close()
        err.append(np.linalg.norm(rho[1] - rho[0]) / np.linalg.norm(rho[0]))
    mean = float(np.exp(np.mean(np.log(err))))
    assert mean < 1.9e-8, mean

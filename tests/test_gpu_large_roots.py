"""Roots beyond the shared memory with fewer tiles than CTAs: the tiles are planned and refused,
then the tensor cores (TF32X3, BF16X3) or a second tile plan (FP32) takes the exponential.

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


@pytest.mark.parametrize("D", [17, 20])
def test_root_of_three_chains_matches_the_oracle_in_every_mode(D):
    p = W.singlet_fission(seed=13, n_env=3, L=2, d=6, D=D, n_modes=6, dt=0.5, n_steps=1)
    o = TTNS(p)
    o.step(p.dt)
    for prec in (ttns.TTNS_FP32, ttns.TTNS_TF32X3, ttns.TTNS_BF16X3, ttns.TTNS_FP64):
        g = ttns.Tree(p, precision=prec)
        g.step(p.dt, 1)
        tol = 1e-7 if prec == ttns.TTNS_FP64 else 1e-6
        assert np.abs(g.rho() - o.rho_el()).max() < tol, prec
        np.testing.assert_allclose(g.occupations(), o.occupations(), atol=10 * tol)
        g.close()

"""The FP64 sweep keeps the norm to rounding.

A step of a one-site chain has six exponentials, four QRs and four absorbs, each of which leaves
the norm as it is up to about two roundings (of eps = 2^-52) of its own: 2 sqrt(14) eps added at
random, taken as 8 eps for the root mean square over many step sizes.  Bessel coefficients that carry
the rounding of every order before them are off by some twenty eps each at these arguments (1 to 6):
over 20 eps a step.
"""
import numpy as np
import pytest

from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def test_a_step_keeps_the_norm_to_rounding():
    dev = []
    for dt in np.linspace(8.0, 30.0, 64):
        p = W.spin_boson(L=1, d=8, D=2, omega_c=0.05, alpha=0.2, dt=float(dt))
        g = ttns.Tree(p, precision=ttns.TTNS_FP64)
        g.step(p.dt, 1)
        dev.append(g.observables()[0] - 1.0)
        g.close()
    rms = float(np.sqrt(np.mean(np.square(dev))))
    assert rms < 8 * 2.0 ** -52, rms / 2.0 ** -52

"""State files of another problem of the same shape: ttns_load_state takes the file's operators with
its state, so that the run goes on as the file's own run, bit for bit, also where the entries of
its sparse operators are in other columns than those of the tree that it is loaded into.
"""
import struct

import numpy as np
import pytest

from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _problem(pairs, n_env=1, seed=0):
    """Five states with a diagonal H_S; every chain couples the given pairs of states."""
    rng = np.random.default_rng(seed)
    Wb = np.zeros((5, 5), dtype=complex)
    for i, j in pairs:
        Wb[i, j] = Wb[j, i] = rng.uniform(0.3, 1.0)
    w = np.linspace(0.05, 0.2, 8)
    envs = [W.Environment(W_bar=Wb, spectral=("modes", w, 0.2 * w), L=3, d=4, D=5) for _ in range(n_env)]
    return W.Problem(name="pairs", H_S=np.diag(rng.uniform(1.5, 2.5, 5)).astype(complex), envs=envs, dt=0.5, n_steps=4,
                     psi_el=np.full(5, 5 ** -0.5, dtype=complex))


@pytest.mark.parametrize("prec", [ttns.TTNS_FP64, ttns.TTNS_TF32X3])
@pytest.mark.parametrize("n_env,kw", [(1, dict(cluster_ctas=16)), (1, dict(cluster_ctas=1)), (2, dict(cluster_ctas=8)),
                                      (2, dict(grid_threshold=1))])
def test_load_state_takes_the_sparse_operators_of_the_file(tmp_path, n_env, kw, prec):
    pa, pb = _problem([(0, 1), (2, 3)], n_env, 1), _problem([(0, 2), (1, 4)], n_env, 2)
    path = str(tmp_path / "b.ck")
    b = ttns.Tree(pb, precision=prec, **kw)
    b.step(pb.dt, 2)
    b.save(path)
    b.step(pb.dt, 2)
    a = ttns.Tree(pa, precision=prec, **kw)
    a.step(pa.dt, 1)
    a.load_state(path)
    a.step(pb.dt, 2)
    assert np.array_equal(a.rho(), b.rho()) and np.array_equal(a.occupations(), b.occupations())
    a.close()
    b.close()


def test_a_column_out_of_range_is_refused(tmp_path):
    pb = _problem([(0, 2), (1, 4)])
    path = str(tmp_path / "bad.ck")
    b = ttns.Tree(pb)
    b.step(pb.dt, 1)
    b.save(path)
    data = bytearray(open(path, "rb").read())
    cols = b"".join(struct.pack("<dd", float(c), 0.0) for c in (2, 4, 0, 0, 1))  # the coupling's table (row 3 is empty)
    at = data.find(cols)
    assert at > 0 and data.find(cols, at + 1) < 0
    data[at:at + 8] = struct.pack("<d", 5.0)
    open(path, "wb").write(bytes(data))
    rho = b.rho()
    with pytest.raises(ttns.TTNSError) as e:
        b.load_state(path)
    assert e.value.code == 7
    assert np.array_equal(b.rho(), rho)  # the state is as it was
    b.close()

"""The forms that the sweep chooses between by size (site plans, resident and element-wise
exponentials, tiled products, projections over rows, one or two CTAs per SM, split layer
products), each at the sizes where it can go wrong, against the FP64 CPU oracle.

Tolerances: populations and density matrices as in test_gpu_parity.py, 1e-7 in FP64 and 1e-6 in
the mixed modes (a few steps of trees whose QR cutoff does not steer the result).  A layer
product with FP32-level operands is off by the dropped low x low terms (2^-22 of sum |a b|) and
one FP32 rounding per K step of 32 (2^-24 each): 4e-6 covers K up to 1600.
"""
import numpy as np
import pytest

from oracle.ttns import TTNS
from paper_1710_01362_gb300 import build, ttns
from paper_1710_01362_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {ttns.TTNS_FP64: 1e-7, ttns.TTNS_TF32X3: 1e-6, ttns.TTNS_BF16X3: 1e-6}


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _oracle(p, n):
    o = TTNS(p)
    for _ in range(n):
        o.step(p.dt)
    return o


# (problem, options): fewer rows than CTAs, odd and even bonds, one leg of dimension 1, Fock legs
# longer and shorter than the bonds, a root with two legs, null columns in runs
SITES = {
    "two_leg_root_D1": (lambda: W.spin_boson(L=3, d=4, D=1), {}),
    "rows_below_ctas": (lambda: W.spin_boson(L=6, d=3, D=3), dict(cluster_ctas=16)),
    "odd_17x5": (lambda: W.sf_small(seed=3, n_env=2, L=4, d=5, D=17, n_modes=8), {}),
    "even_16x4_two_ctas": (lambda: W.sf_small(seed=4, n_env=2, L=4, d=4, D=16, n_modes=8), dict(cluster_ctas=2)),
    "long_fock_leg": (lambda: W.spin_boson(L=3, d=31, D=5), dict(cluster_ctas=8)),
    "grid_team": (lambda: W.sf_small(seed=5, n_env=3, L=3, d=7, D=9, n_modes=8), dict(grid_threshold=1)),
    "er_one_cta": (lambda: W.sf_small(seed=6, n_env=4, L=3, d=4, D=6, n_modes=8, er_tree=True, D_er=7),
                   dict(cluster_ctas=1)),
}


@pytest.mark.parametrize("name", list(SITES))
def test_site_and_resident_forms_match_the_oracle(name):
    make, kw = SITES[name]
    p = make()
    o = _oracle(p, 3)
    for prec, tol in TOL.items():
        g = ttns.Tree(p, precision=prec, **kw)
        g.step(p.dt, 3)
        assert np.abs(g.rho() - o.rho_el()).max() < tol, prec
        np.testing.assert_allclose(g.occupations(), o.occupations(), atol=10 * tol)
        if prec == ttns.TTNS_FP64:  # bond spectra: matrices of every size in one batch
            np.testing.assert_allclose(g.bond_entropies(), o.bond_entropies(), atol=1e-6)
        g.close()


@pytest.mark.parametrize("D", [13, 17, 21])
def test_large_star_root_matches_the_oracle(D):
    # root of D^4 x 5 on the whole grid: tiles of 5 D^2 elements, each block shape of the fibre
    # products, odd remainders; environment projections over rows
    p = W.singlet_fission(seed=11, n_env=4, L=2, d=5, D=D, n_modes=6, dt=0.5, n_steps=1)
    o = _oracle(p, 1)
    for prec in (ttns.TTNS_FP64, ttns.TTNS_TF32X3):
        g = ttns.Tree(p, precision=prec)
        g.step(p.dt, 1)
        assert np.abs(g.rho() - o.rho_el()).max() < TOL[prec], prec
        np.testing.assert_allclose(g.occupations(), o.occupations(), atol=10 * TOL[prec])
        g.close()


@pytest.mark.parametrize("ctas,n", [(1, 304), (2, 160)])
def test_sets_of_small_trees_equal_the_oracle_on_one_or_two_ctas_per_sm(ctas, n):
    ps = [W.sf_small(seed=100 + k, n_env=2, L=2, d=3, D=3 + k % 3, n_modes=4) for k in range(n)]
    pick = [0, 1, n // 2, n - 1]
    ref = {k: _oracle(ps[k], 2).populations() for k in pick}
    for prec in (ttns.TTNS_FP64, ttns.TTNS_TF32X3):
        pops = []
        for grid in (0, 152):  # as many CTAs as fit, two per SM; at most one per SM
            g = ttns.Tree(ps, precision=prec, cluster_ctas=ctas, grid_ctas=grid)
            g.step(ps[0].dt, 1)
            g.step(ps[0].dt, 1)
            pops.append(np.array([g.populations(k) for k in range(n)]))
            g.close()
        assert np.abs(pops[0] - pops[1]).max() < TOL[prec]
        for k in pick:
            assert np.abs(pops[0][k] - ref[k]).max() < TOL[prec], k


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (129, 31, 33), (33, 65, 257), (64, 129, 1025)])
def test_layer_products_at_tile_and_split_edges(M, N, K):
    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((M, K)).astype(np.float32)
    B = rng.standard_normal((K, N)).astype(np.float32)
    Ad, Bd = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    C = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    code = ttns.lib().ttns_mlp_gemm(1, M, N, K, Ad.data_ptr(), K, 0, Bd.data_ptr(), N, 0, C.data_ptr(), N, 0, None, None)
    assert code == 0, ttns.lib().ttns_last_error()
    torch.cuda.synchronize()
    A, B = A.astype(np.float64), B.astype(np.float64)
    assert (np.abs(C.double().cpu().numpy() - A @ B) / (np.abs(A) @ np.abs(B))).max() < 4e-6

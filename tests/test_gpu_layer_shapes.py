"""Layer products whose row or column tiles exceed the 65535 that a grid's second dimension holds.

With one term per output the product of FP32-level operands is off by the dropped low x low term
and the tensor core's rounding, 2^-22 and 2^-23 of it: 1e-6.
"""
import numpy as np
import pytest

from paper_1710_01362_gb300 import build, ttns

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("kind,tol", [(1, 1e-6), (3, 2.0 ** -7)])
@pytest.mark.parametrize("M,N", [(1, 64 * 65535 + 70), (128 * 65536 + 5, 3)])
def test_products_of_very_many_tiles(M, N, kind, tol):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.rand((M, 1), generator=g, device="cuda") + 0.5
    B = torch.rand((1, N), generator=g, device="cuda") + 0.5
    C = torch.zeros((M, N), device="cuda")
    code = ttns.lib().ttns_mlp_gemm(kind, M, N, 1, A.data_ptr(), 1, 0, B.data_ptr(), N, 0, C.data_ptr(), N, 0, None, None)
    assert code == 0, ttns.lib().ttns_last_error()
    ref = A.double() * B.double()
    assert ((C.double() - ref).abs() / ref).max().item() < tol

"""The exact-digit GEMM with more output columns than one launch's grid can hold in its
second dimension (65535 blocks of 32): the same bits as narrower products of the same
columns, at the widest single launch, one past it and past the grid's own limit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def omm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2209_05934_gb300 import omm as _omm
    _omm.lib()
    return _omm


def product(omm, A, B, Cin, nd):
    """-2 A B + 4 Cin, column-major device tensors."""
    (M, K), N = A.shape, B.shape[1]
    C = torch.zeros((N, M), dtype=torch.float64, device="cuda").T
    nb = omm.op_exact_gemm_workspace_bytes(M, N, K, nd)
    ws = torch.zeros(nb // 8 + 64, dtype=torch.float64, device="cuda")
    st = omm.op_exact_gemm(0, 0, M, N, K, nd, -2.0, A, M, B, K, 4.0, Cin, M, C, M, ws, nb)
    torch.cuda.synchronize()
    assert st == omm.OK, omm.lib().omm_last_error()
    return C


@pytest.mark.parametrize("nd", [2, 7])
@pytest.mark.parametrize("N", [65280 * 32, 65280 * 32 + 1, 65535 * 32 + 257])
def test_wide_product(omm, N, nd):
    M, K = 3, 8
    g = torch.Generator(device="cuda").manual_seed(N)
    normal = lambda r, c: torch.randn(c, r, generator=g, device="cuda", dtype=torch.float64).T
    A, B, Cin = normal(M, K), normal(K, N), normal(M, N)
    C = product(omm, A, B, Cin, nd)
    for lo, hi in ((0, 5000), (65280 * 32 - 3000, N)):
        cut = lambda X: X[:, lo:hi].T.contiguous().T
        assert torch.equal(C[:, lo:hi], product(omm, A, cut(B), cut(Cin), nd))
    # a row's or column's rounding is at most 2^-(7 nd) of its largest element's power of
    # two, twice that element at most, and level nd + 2 on is left out
    bound = 8.0 * K * 2.0 ** -(7 * nd - 6) * A.abs().amax(1)[:, None] * B.abs().amax(0)[None, :]
    ref = -2.0 * (A @ B) + 4.0 * Cin
    assert bool(((C - ref).abs() <= bound + 1e-13 * (ref.abs() + 1)).all())

"""Memory of the FP64 products' residue planes: one size for the library's allocation and the
server's admission, S's half left out where S = I."""
import pytest


@pytest.fixture(scope="module")
def omm():
    import __graft_entry__ as g
    g.build()
    from paper_2209_05934_gb300 import omm as _omm
    _omm.lib()
    return _omm


def planes(m, n, hs_rows, precon):
    """19 BF16 planes of every operand and a byte of each per output, 256-byte aligned parts."""
    up, k, k2 = (lambda v: -(-v // 256) * 256), -(-m // 8) * 8, -(-2 * n // 8) * 8
    rows = [hs_rows * k, 2 * n * k, 2 * n * k, m * k2, n * k2] + ([m * k, n * k] if precon else [0, 0])
    words = lambda M, N: 19 * (-(-N // 4)) * (-(-M // 4) * 4)
    return (sum(up(2 * 19 * r) for r in rows) + up(4 * (4 * m + 6 * n + 1)) + up(8 * 32 * m)
            + up(4 * max(2 * words(m, n), words(2 * n, 2 * n))))


@pytest.mark.parametrize("m,n", [(8, 2), (129, 65), (2048, 512)])
@pytest.mark.parametrize("cholesky,precon", [(0, 0), (1, 0), (0, 1)])
def test_size_counts_what_the_products_read(omm, m, n, cholesky, precon):
    from paper_2209_05934_gb300 import serving
    want = planes(m, n, m if cholesky else 2 * m, precon)
    assert omm.product_planes_bytes(m, n, cholesky, precon) == want
    arrays = serving.footprint_bytes(m, n, omm.PREC_FP64, cholesky=cholesky, precon=precon) - want
    assert arrays == 8 * (2 * m * m + 8 * m * n + 6 * n * n)


def test_refused_sizes(omm):
    assert omm.product_planes_bytes(0, 1) == -1 and omm.product_planes_bytes(4, 5) == -1


@pytest.mark.gpu
@pytest.mark.parametrize("cholesky", [0, 1])
def test_create_takes_that_much(omm, cholesky):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m, n = 4096, 1024
    used = {}
    for form in (omm.FP64_CUDA_CORES, omm.FP64_RESIDUES):
        free = torch.cuda.mem_get_info()[0]
        s = omm.Solver(m, n, 8, cholesky=cholesky, fp64_products=form)
        used[form] = free - torch.cuda.mem_get_info()[0]
        s.close()
    more = used[omm.FP64_RESIDUES] - used[omm.FP64_CUDA_CORES]
    assert abs(more - omm.product_planes_bytes(m, n, cholesky)) <= 32 << 20

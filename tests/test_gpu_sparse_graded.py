"""The FP64 linear-scaling form on graded operands: orbitals shifted far up in H and
coefficients that are small against them, and orbitals whose overlap is between tails.

Every output is held to the bound of an FP64 multiply-add chain, element by element:
with K terms, |error| <= (K + 2) 2^-53 sum |a_k| |b_k|, whatever the sizes of the other
elements of the row and the column."""
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


def to_dense(rp, col, vals, nr, nc, br, bc):
    A = np.zeros((nr * br, nc * bc))
    for I in range(nr):
        for b in range(rp[I], rp[I + 1]):
            A[I * br:(I + 1) * br, col[b] * bc:(col[b] + 1) * bc] = vals[b]
    return A


def check(got, A, B, what, symmetrised=False):
    q = np.longdouble
    ref = A.astype(q) @ B.astype(q)
    bound = ((A != 0).astype(float) @ (B != 0).astype(float) + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(B))
    if symmetrised:          # the start keeps (X + X^T) / 2
        ref = (ref + ref.T) / 2
        bound = (bound + bound.T) / 2 + 2.0 ** -52 * np.abs(ref).astype(float)
    err = np.abs((got - ref).astype(float))
    assert (err <= bound).all(), (what, float((err / np.where(bound > 0, bound, 1)).max()))


@pytest.mark.parametrize("shift,decay", [(1.0, 0.0), (1e3, 0.0), (1e9, 0.0), (1.0, 3.0), (1e6, 3.0)])
def test_products_hold_the_fp64_bound_element_by_element(omm, shift, decay):
    import synth
    s0_ = synth.make_system(4, 3, 2, seed=5)
    hrp, hcol, Hv, Sv = s0_.bsr()
    wrp, wcol = s0_.w_pattern(6.0)
    N, m, n = s0_.natoms, s0_.m, s0_.n
    rows = np.repeat(np.arange(N), np.diff(hrp))
    wrows = np.repeat(np.arange(N), np.diff(wrp))
    Hv, W0 = Hv.copy(), np.random.default_rng(9).standard_normal((len(wcol), 8, 2))
    Hv[rows == hcol, 3, 3] += shift                       # the fourth orbital of every atom
    W0[:, 3, :] /= shift
    r = np.linalg.norm(s0_.positions[wrows] - s0_.positions[wcol], axis=1)
    W0 *= np.exp(-decay * r)[:, None, None]               # from its own atom outwards
    s = omm.SparseSolver(m, n, 8, 2, hrp, hcol, wrp, wcol, eta_auto=0, eta=0.0, max_iter=0, filter_eps=0.0)
    s.set_HS(np.ascontiguousarray(Hv), np.ascontiguousarray(Sv))
    s.solve(np.ascontiguousarray(W0), tol=1e-14, raise_on_error=False)
    got = {k: s.get_array(k) for k in (omm.ARRAY_HW, omm.ARRAY_SW, omm.ARRAY_HW_N, omm.ARRAY_SW_N)}
    hw, nn = s.get_pattern(omm.PATTERN_HW), s.get_pattern(omm.PATTERN_N)
    s.close()
    H, S = (to_dense(hrp, hcol, v, N, N, 8, 8) for v in (Hv, Sv))
    W = to_dense(wrp, wcol, W0, N, N, 8, 2)
    dn = lambda k, pat, br: to_dense(*pat, got[k].reshape(-1, br, 2), N, N, br, 2)
    HW, SW = dn(omm.ARRAY_HW, hw, 8), dn(omm.ARRAY_SW, hw, 8)
    check(HW, H, W, "H'W")
    check(SW, S, W, "S W")
    check(dn(omm.ARRAY_HW_N, nn, 2), W.T, HW, "W^T H'W", True)
    check(dn(omm.ARRAY_SW_N, nn, 2), W.T, SW, "W^T S W", True)

"""The dense FP64 form on graded operands: orbitals shifted far up in H with coefficients
that are small against them, decaying rows against decaying columns, energies in large
and in small units, coefficients near the bottom of the FP64 range.

Every product is held to the bound of an FP64 multiply-add chain, element by element: with
K terms, |error| <= (K + 2) 2^-53 sum |a_k| |b_k| (and 2^-1074 a term where it underflows),
whatever the sizes of the other elements of the row and the column."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

U, TINY = 2.0 ** -53, 2.0 ** -1074


@pytest.fixture(scope="module")
def omm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2209_05934_gb300 import omm as _omm
    _omm.lib()
    return _omm


def dev(a):
    return torch.from_numpy(np.asfortranarray(a)).to("cuda")


def problem(kind, x, m, n):
    rng = np.random.default_rng(m + n)
    A = rng.standard_normal((m, m))
    H, W = A + A.T, rng.standard_normal((m, n))
    B = rng.uniform(-1, 1, (m, m)) * (0.2 / m)
    S = np.eye(m) + B + B.T
    i, j = np.arange(m), np.arange(n) * m / n
    if kind == "unit":
        H *= x
    elif kind == "shift":            # every 16th orbital x above the others
        H[i[::16], i[::16]] += x
        W[::16] /= x
    elif kind == "decay":            # x: decay per row
        near = np.exp(-x * np.abs(i[:, None] - i[None, :]))
        H, S = H * near, S * near
        W *= np.exp(-x * np.abs(i[:, None] - j[None, :]))
    elif kind == "tiny":
        W *= x
    return H, S, W


def check(got, A, B, what, symmetrised=False):
    q = np.longdouble
    ref = A.astype(q) @ B.astype(q)
    bound = (A.shape[1] + 2) * (U * (np.abs(A) @ np.abs(B)) + TINY)
    if symmetrised:                  # the start keeps (X + X^T) / 2
        ref = (ref + ref.T) / 2
        bound = (bound + bound.T) / 2 + 2 * U * np.abs(ref).astype(float)
    err = np.abs((got - ref).astype(float))
    assert (err <= bound).all(), (what, float((err / np.where(bound > 0, bound, 1)).max()))


@pytest.mark.parametrize("m,n", [(33, 5), (130, 33), (257, 130)])
@pytest.mark.parametrize("kind,x", [("unit", 1e-18), ("unit", 2e5), ("unit", 1e30), ("shift", 1e3), ("shift", 1e9),
                                    ("decay", 0.02), ("decay", 0.5), ("decay", 3.0), ("tiny", 1e-300)])
def test_products_hold_the_fp64_bound_element_by_element(omm, kind, x, m, n):
    H, S, W = problem(kind, x, m, n)
    got = {}
    for steps in (0, 1):
        s = omm.Solver(m, n, 8, eta_auto=0, eta=0.0, max_iter=steps)
        s.set_HS(dev(H), dev(S))
        s.solve(dev(W), tol=1e-10, raise_on_error=False)
        got[steps] = {k: s.get_array(k) for k in (omm.ARRAY_HW, omm.ARRAY_SW, omm.ARRAY_HW_N, omm.ARRAY_SW_N,
                                                  omm.ARRAY_G)}
        s.close()
    HW, SW, h0, s0 = (got[0][k] for k in (omm.ARRAY_HW, omm.ARRAY_SW, omm.ARRAY_HW_N, omm.ARRAY_SW_N))
    G = got[1][omm.ARRAY_G]
    check(HW, H, W, "H'W")
    check(SW, S, W, "S W")
    check(h0, W.T, HW, "W^T H'W", True)
    check(s0, W.T, SW, "W^T S W", True)
    q = np.longdouble
    ref = 4 * HW.astype(q) - 2 * (SW.astype(q) @ h0.astype(q) + HW.astype(q) @ s0.astype(q))
    bound = (2 * (2 * n + 2) * (U * (np.abs(SW) @ np.abs(h0) + np.abs(HW) @ np.abs(s0)) + TINY)
             + 4 * U * (4 * np.abs(HW) + np.abs(ref).astype(float)))
    err = np.abs((G - ref).astype(float))
    assert (err <= bound).all(), ("G", float((err / np.where(bound > 0, bound, 1)).max()))

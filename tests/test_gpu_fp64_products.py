"""The FP64 form's products through residue planes (tensor cores): H'W, SW, W^T(..)
and the gradient at sizes around the tiles (128 and 256 rows, 256 columns), the
1024-long exact pieces of K and odd sizes, on rows and columns whose scales spread
over many orders of magnitude, against products in extended precision.

max_iter = 0 leaves the solve at its start: W is W0 and the arrays hold the first
products; the gradient of that start is what one step (max_iter = 1) leaves in G.  The operands' fixed-point rounding is 2^-62 of ||a|| ||b|| each, at most
doubled by each power-of-two row scale, so an inner product is within
2^-58 ||a|| ||b|| and the rounding of the result to FP64."""
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


def dev(a):
    return torch.from_numpy(np.asfortranarray(a)).to("cuda")


def problem(m, n, spread, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((m, m)) * np.exp(rng.uniform(-spread, spread, (m, 1)))
    H = A + A.T
    B = rng.uniform(-1, 1, (m, m)) * (0.2 / m)
    S = np.eye(m) + B + B.T
    W = rng.standard_normal((m, n)) * np.exp(rng.uniform(-spread, spread, (1, n)))
    W[:, 0] = 0.0                     # a zero column
    return H, S, W


def check(got, A, B, what):
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    bound = (2.0 ** -58 * np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
             + 2.0 ** -52 * np.abs(ref).astype(float))
    err = np.abs((got - ref).astype(float))
    assert (err <= bound).all(), (what, float((err / np.where(bound > 0, bound, 1)).max()))


@pytest.mark.parametrize("m,n,spread", [(8, 2, 0.0), (65, 33, 0.0), (128, 32, 2.0), (129, 65, 2.0), (257, 127, 0.0),
                                        (512, 258, 3.0), (1024, 31, 0.0), (1031, 17, 2.0), (2051, 5, 0.0)])
def test_products_match_extended_precision(omm, m, n, spread):
    H, S, W = problem(m, n, spread, m + n)
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
    check(h0, W.T, HW, "W^T H'W")
    check(s0, W.T, SW, "W^T S W")
    left, right = np.hstack([SW, HW]), np.vstack([h0, s0])
    ref = 4 * HW.astype(np.longdouble) - 2 * (left.astype(np.longdouble) @ right.astype(np.longdouble))
    bound = (2.0 ** -57 * np.linalg.norm(left, axis=1)[:, None] * np.linalg.norm(right, axis=0)[None, :]
             + 2.0 ** -51 * (4 * np.abs(HW) + np.abs(ref).astype(float)))
    assert (np.abs((G - ref).astype(float)) <= bound).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_ends_the_solve(omm, bad):
    H, S, W = problem(130, 20, 0.0, 3)
    W[7, 3] = bad
    s = omm.Solver(130, 20, 8, eta_auto=0, eta=0.0)
    s.set_HS(dev(H), dev(S))
    E, it, st = s.solve(dev(W), tol=1e-10, raise_on_error=False)
    s.close()
    assert st == omm.ERR_NONFINITE

"""The FP64 gathers of the linear-scaling form in fixed-point integers: H'W, SW,
W^T(..) and the gradient of small systems against dense products in extended
precision, with rows and columns whose scales spread over orders of magnitude, a zero
column and patterns down to a single block.

Operands are rounded to 57 bits of their rows' and columns' norms; with both power-of-two
scales a factor of four off at most, eight standard deviations of the rounding of an
inner product are 2^-51 ||a|| ||b||."""
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


def check(got, A, B, mask, what):
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    bound = (2.0 ** -51 * np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
             + 2.0 ** -52 * np.abs(ref).astype(float))
    err = np.abs((got - ref).astype(float)) * mask
    assert (err <= bound).all(), (what, float((err / np.where(bound > 0, bound, 1)).max()))


@pytest.mark.parametrize("dims,radius,spread", [((1, 1, 1), 3.0, 0.0), ((2, 2, 1), 3.0, 2.0), ((3, 3, 2), 4.5, 3.0),
                                                ((4, 4, 4), 6.0, 0.0)])
def test_gathers_match_extended_precision(omm, dims, radius, spread):
    import synth
    s0_ = synth.make_system(*dims, seed=sum(dims))
    hrp, hcol, Hv, Sv = s0_.bsr()
    wrp, wcol = s0_.w_pattern(radius)
    N, m, n = s0_.natoms, s0_.m, s0_.n
    rng = np.random.default_rng(N)
    scale = np.exp(rng.uniform(-spread, spread, N))            # per atom: H rows and columns
    rows = np.repeat(np.arange(N), np.diff(hrp))
    Hv = Hv * (scale[rows] * scale[hcol])[:, None, None]
    W0 = rng.standard_normal((len(wcol), 8, 2)) * np.exp(rng.uniform(-spread, spread, N))[wcol][:, None, None]
    W0[wcol == 0, :, 1] = 0.0                                  # a zero column
    got = {}
    for steps in (0, 1):
        s = omm.SparseSolver(m, n, 8, 2, hrp, hcol, wrp, wcol, eta_auto=0, eta=0.0, max_iter=steps)
        s.set_HS(np.ascontiguousarray(Hv), np.ascontiguousarray(Sv))
        s.solve(np.ascontiguousarray(W0), tol=1e-14, raise_on_error=False)
        got[steps] = {k: s.get_array(k) for k in range(7)}
        hw, nn = s.get_pattern(omm.PATTERN_HW), s.get_pattern(omm.PATTERN_N)
        s.close()
    H, S = (to_dense(hrp, hcol, v, N, N, 8, 8) for v in (Hv, Sv))
    W = to_dense(wrp, wcol, W0, N, N, 8, 2)
    dn = lambda k, pat, r, br: to_dense(*pat, got[0][k].reshape(-1, br, 2), r, N, br, 2)
    HW, SW = dn(omm.ARRAY_HW, hw, N, 8), dn(omm.ARRAY_SW, hw, N, 8)
    h0, sn = dn(omm.ARRAY_HW_N, nn, N, 2), dn(omm.ARRAY_SW_N, nn, N, 2)
    check(HW, H, W, 1, "H'W")
    check(SW, S, W, 1, "S W")
    check(h0, W.T, HW, 1, "W^T H'W")
    check(sn, W.T, SW, 1, "W^T S W")
    # the gradient of the start, which one step leaves in G, on the pattern of W
    mask = to_dense(wrp, wcol, np.ones((len(wcol), 8, 2)), N, N, 8, 2)
    G = to_dense(wrp, wcol, got[1][omm.ARRAY_G].reshape(-1, 8, 2), N, N, 8, 2)
    q = np.longdouble
    ref = 2 * (2 * HW.astype(q) - SW.astype(q) @ h0.astype(q) - HW.astype(q) @ sn.astype(q))
    nrm = lambda A, B: np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
    bound = 2.0 ** -50 * (nrm(SW, h0) + nrm(HW, sn)) + 2.0 ** -50 * np.abs(HW)
    assert (np.abs((G - ref).astype(float)) * mask <= bound).all()


def test_nonfinite_block_ends_the_solve(omm):
    import synth
    s0_ = synth.make_system(2, 2, 2, seed=4)
    hrp, hcol, Hv, Sv = s0_.bsr()
    wrp, wcol = s0_.w_pattern(4.0)
    W0 = np.random.default_rng(1).standard_normal((len(wcol), 8, 2))
    W0[3, 2, 1] = np.inf
    s = omm.SparseSolver(s0_.m, s0_.n, 8, 2, hrp, hcol, wrp, wcol, eta_auto=0, eta=0.0)
    s.set_HS(Hv, Sv)
    E, it, st = s.solve(W0, tol=1e-10, raise_on_error=False)
    s.close()
    assert st == omm.ERR_NONFINITE

"""Where the products of dense FP64 handles run: the CUDA-core form through the same
dense, Cholesky and preconditioned solves as the residue form, and the form reported, also
where there is no memory for the residue form."""
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


def system(atoms, seed=1, drop=0):
    import synth
    s = synth.make_system(*atoms, seed=seed)
    keep = s.m - drop
    H, S = s.dense_H()[:keep, :keep], s.dense_S()[:keep, :keep]
    W0 = np.random.default_rng(seed).standard_normal((keep, s.n)) / np.sqrt(keep)
    return s, H, S, W0


def solved(omm, H, S, W0, T=None, **opts):
    m, n = W0.shape
    s = omm.Solver(m, n, 8, **opts)
    assert s.product_form() == omm.PRODUCTS_NONE
    s.set_HS(dev(H), dev(S))
    if T is not None:
        s.set_T(dev(T))
    E, it, _ = s.solve(dev(W0), tol=1e-12)
    d, form = s.diag(), s.product_form()
    rho = s.get_density()
    s.close()
    return E, d.orth, rho, form


@pytest.mark.parametrize("atoms,drop", [((2, 1, 1), 0), ((2, 2, 2), 3), ((4, 4, 2), 0)])
@pytest.mark.parametrize("variant", ["plain", "cholesky", "precon"])
def test_cuda_core_products_reach_the_same_solution(omm, atoms, drop, variant):
    sy, H, S, W0 = system(atoms, drop=drop)
    T, opts = None, {}
    if variant == "cholesky":
        opts = dict(cholesky=1)
    elif variant == "precon":
        T = sy.dense_T()[:len(H), :len(H)]
        H, opts = H + T, dict(precon=-1)
    E0, o0, r0, f0 = solved(omm, H, S, W0, T, fp64_products=omm.FP64_RESIDUES, **opts)
    E1, o1, r1, f1 = solved(omm, H, S, W0, T, fp64_products=omm.FP64_CUDA_CORES, **opts)
    assert (f0, f1) == (omm.PRODUCTS_RESIDUES, omm.PRODUCTS_CUDA_CORES)
    # two solves to RelTol 1e-12: the energy's error is second order in W's, rho's first order
    assert abs(E0 - E1) <= 1e-10 * abs(E0)
    np.testing.assert_allclose(r1, r0, rtol=0, atol=1e-4)
    assert o0 < 1e-3 and o1 < 1e-3


def test_without_memory_a_solve_reports_or_refuses(omm):
    _, H, S, W0 = system((4, 4, 4))
    m, n = W0.shape
    E2, _, _, _ = solved(omm, H, S, W0, fp64_products=omm.FP64_CUDA_CORES)
    w0 = dev(W0)
    torch.cuda.empty_cache()
    # room for the arrays, but not for planes beside what the driver is left with (256 MB)
    fill = torch.empty(max(torch.cuda.mem_get_info()[0] - (200 << 20), 0), dtype=torch.uint8, device="cuda")
    res = omm.Solver(m, n, 8, fp64_products=omm.FP64_RESIDUES)
    aut = omm.Solver(m, n, 8)
    res.set_HS(dev(H), dev(S))
    aut.set_HS(dev(H), dev(S))
    E1, _, _ = aut.solve(w0, tol=1e-12)
    assert aut.product_form() == omm.PRODUCTS_CUDA_CORES
    with pytest.raises(omm.OmmError) as err:
        res.solve(w0, tol=1e-12)
    assert err.value.status == omm.ERR_NOMEM
    del fill
    torch.cuda.empty_cache()
    E0, _, _ = res.solve(w0, tol=1e-12)                    # with memory again
    assert res.product_form() == omm.PRODUCTS_RESIDUES
    E3, _, _ = aut.solve(w0, tol=1e-12)                    # the other form, after graphs of the first
    assert aut.product_form() == omm.PRODUCTS_RESIDUES
    assert E1 == E2 and E3 == E0 and abs(E0 - E1) <= 1e-10 * abs(E0)
    aut.close()
    res.close()

"""The memory of the residue planes of dense FP64 handles: it gives way to the arrays of
other handles and keeps to its share of the device's."""
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


def test_other_handles_get_the_memory_of_idle_planes(omm):
    _, H, S, W0 = system((8, 4, 4))
    m, n = W0.shape
    a = omm.Solver(m, n, 8)
    a.set_HS(dev(H), dev(S))
    Wa = torch.empty((n, m), dtype=torch.float64, device="cuda").T
    first = a.solve(dev(W0), tol=1e-10, W_out=Wa)
    Wa = Wa.clone()
    # leave less than a second handle's arrays need, but not less than that and a's planes
    big_m, big_n = 2048, 512
    need = 8 * (2 * big_m ** 2 + 10 * big_m * big_n + 6 * big_n ** 2)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(max(free - need + (4 << 20), 0), dtype=torch.uint8, device="cuda")
    left = torch.cuda.mem_get_info()[0]
    assert left < need < left + 38 * 2 * m * m
    b = omm.Solver(big_m, big_n, 8)
    b.close()
    del fill
    torch.cuda.empty_cache()
    # a takes its planes again and repeats its solve bit for bit
    Wb = torch.empty((n, m), dtype=torch.float64, device="cuda").T
    again = a.solve(dev(W0), tol=1e-10, W_out=Wb)
    assert first == again and torch.equal(Wa, Wb)
    a.close()


@pytest.mark.parametrize("short", [False, True])
def test_planes_of_all_handles_beyond_an_eighth_of_the_device(omm, short):
    """With room all eight handles hold planes (57 GB); where they would leave less than a
    quarter of the device free, those of the handles not in use keep below an eighth."""
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    m, n = 7000, 1750
    arrays = 8 * (2 * m * m + 8 * m * n + 6 * n * n)
    planes = 38 * (2 * m * m + 6 * m * n + 2 * n * n)
    count, slack = 8, 8 * (64 << 20)
    fill = torch.empty(max(free - int(0.3 * total), 0) if short else 0, dtype=torch.uint8, device="cuda")
    free = torch.cuda.mem_get_info()[0]
    hs = [omm.Solver(m, n, 8) for _ in range(count)]
    used = free - torch.cuda.mem_get_info()[0]
    for s in hs:
        s.close()
    left = free - torch.cuda.mem_get_info()[0]
    del fill
    torch.cuda.empty_cache()
    if short:
        assert used <= count * arrays + total // 8 + slack
    else:
        assert used >= count * (arrays + planes)
    assert left <= slack

"""What orders a kernel's reads with the launches before it.  Solves launched
kernel by kernel (profiling) against the same solves replayed from captured
graphs, bit for bit: the values a kernel reads must be those of the launches
before it on either path."""
import numpy as np
import pytest

from paper_1905_08717_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_08717_gb300 import build
    build.build()


@pytest.mark.parametrize("rk,prec", [(2, I.PREC_FP64), (3, I.PREC_FP64), (3, I.PREC_MIXED)])
def test_one_level_tree_takes_the_step_of_its_macro_step(rk, prec):
    """min_level == max_level with adaptation on and node arrays beyond those
    that are always kept whole: the head of a macro step holds the only launch
    before its first stage, so the stage follows directly on the launch that
    sets the fine step, here another one in every macro step."""
    import paper_1905_08717_gb300 as pkg
    p, q = I.euler_2d_quadrants(L=9, min_level=9, rk_order=rk)
    p = p.replace(precision=prec)
    a, b = pkg.Solver(p, q), pkg.Solver(p, q)
    assert b.stats()["device_bytes"] > 32 << 20
    b.profile(True)
    for k in range(6):
        dt = 1e-4 * (1.0 + 0.5 * (-1) ** k)
        for s in (a, b):
            assert s.iterate(dt, 1) == 1
        (ka, va), (kb, vb) = a.leaves(), b.leaves()
        assert len(ka) == 1 << 18 and np.array_equal(ka, kb)
        assert np.array_equal(va, vb), k
    a.close()
    b.close()


def _problem(dim, eq, L, lb, mode, rk):
    if eq == I.EQ_EULER:
        p, q = (I.euler_2d_quadrants if dim == 2 else I.euler_3d_blast)(L=L, min_level=lb)
    else:
        p = I.Problem(dim=dim, equation=I.EQ_BURGERS, max_level=L, min_level=lb, eps=1e-2)
        x = (np.arange(1 << L) + 0.5) / (1 << L)
        g = np.meshgrid(*([x] * dim), indexing="ij")
        q = sum(np.sin(2 * np.pi * (k + 1) * a + k) for k, a in enumerate(g))[None] * 0.5
    return p.replace(time_mode=mode, rk_order=rk), np.ascontiguousarray(q)


@pytest.mark.parametrize("dim,eq,L,lb,mode,rk", [
    (1, I.EQ_BURGERS, 10, 2, I.TIME_LT, 3), (1, I.EQ_BURGERS, 14, 8, I.TIME_LT, 2), (1, I.EQ_BURGERS, 9, 4, I.TIME_GTS, 3),
    (2, I.EQ_BURGERS, 8, 3, I.TIME_LT, 2), (2, I.EQ_EULER, 9, 4, I.TIME_LT, 3), (2, I.EQ_EULER, 8, 5, I.TIME_GTS, 2),
    (3, I.EQ_EULER, 6, 3, I.TIME_LT, 3),
])
def test_direct_launches_equal_replayed_pieces(dim, eq, L, lb, mode, rk):
    """whole macro steps from captured pieces (a), single iterations and mixed
    counts launched directly between them (b), everything directly (c): the
    publications of both kinds of launches interleave in b"""
    import paper_1905_08717_gb300 as pkg
    p, q = _problem(dim, eq, L, lb, mode, rk)
    nit = 1 << (L - lb)
    dt = 0.2 / (1 << L) / (12.0 if dim == 3 else 4.0)
    a, b, c = (pkg.Solver(p, q) for _ in range(3))
    c.profile(True)
    for k in range(3):
        a.iterate(dt, nit)
        c.iterate(dt, nit)
        if k == 1:
            b.iterate(dt, nit)
        else:
            for n in (1, nit // 2, nit - 1 - nit // 2):
                if n:
                    b.iterate(dt, n)
    (ka, va), (kb, vb), (kc, vc) = a.leaves(), b.leaves(), c.leaves()
    assert np.array_equal(ka, kb) and np.array_equal(ka, kc)
    assert np.array_equal(va, vb) and np.array_equal(va, vc)
    for s in (a, b, c):
        s.close()


@pytest.mark.parametrize("rk,mode", [(3, I.TIME_LT), (2, I.TIME_LT), (2, I.TIME_GTS)])
def test_macro_step_of_2048_iterations(rk, mode):
    """eleven levels above the coarsest: 128 leads and blocks per macro step,
    against the oracle (the same leaves, values to the parity tolerance of the
    adaptive 1D tests) and against direct launches, bit for bit"""
    import oracle
    import paper_1905_08717_gb300 as pkg
    p, q = I.burgers_1d(L=12, min_level=1, rk_order=rk)
    p = p.replace(time_mode=mode)
    dt = 0.25 / (1 << 12)
    a, b, o = pkg.Solver(p, q), pkg.Solver(p, q), oracle.Oracle(p, q)
    b.profile(True)
    for s in (a, b, o):
        s.iterate(dt, 2048)
    (ka, va), (kb, vb), (ko, vo) = a.leaves(), b.leaves(), o.leaves()
    assert np.array_equal(ka, kb) and np.array_equal(va, vb)
    assert np.array_equal(ka, ko)
    assert np.abs(va - vo).max() <= 1e-12 * np.abs(vo).max()
    a.close()
    b.close()


@pytest.mark.parametrize("n", [31, 32])
def test_batches_on_both_sides_of_waiting_first(n):
    """instances of a batch, below the size from which they wait before every
    lookup and at it, against single solvers, bit for bit"""
    import paper_1905_08717_gb300 as pkg
    probs, qs = I.rd_batch(n=n, levels=(6, 8))
    b = pkg.Batch(probs, qs)
    b.step(0.004)
    for i in range(0, n, 5):
        s = pkg.Solver(probs[i], qs[i])
        s.step(0.004)
        for x, y in zip(s.leaves(), b.instances[i].leaves()):
            assert np.array_equal(x, y), i
        s.close()
    b.close()

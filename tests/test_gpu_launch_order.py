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
